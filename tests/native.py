"""Small libraries that a test compiles against the sources of librtc.so: to set a device
word from the host, or to build a kernel around a copy that never lands."""
import ctypes
import subprocess

from paper_1805_07254_gb300 import _build


def compile_so(tmp_dir, name, source):
    src, so = tmp_dir / f"{name}.cu", tmp_dir / f"{name}.so"
    src.write_text(source)
    r = subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-o", str(so), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))
