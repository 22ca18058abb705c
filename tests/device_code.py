"""Small programs over the headers in csrc/, compiled with nvcc as the library is."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1506_06513_gb300", "csrc")


def _compile(source, out, args):
    import __graft_entry__
    b = __graft_entry__._build_module()
    src = os.path.splitext(str(out))[0] + ".cu"
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", CSRC, src, "-o", str(out), *args], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(out)


def program_output(source, tmp_path, *args):
    """What a host program prints (no device work: it runs without a GPU)."""
    exe = _compile(source, tmp_path / "program.exe", args)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    return r.stdout


def shared_library(source, folder, *args):
    """A shared library of kernels and their C entry points, for ctypes."""
    return _compile(source, folder / "kernels.so", ("-shared", "-cudart", "static", *args))
