"""Test libraries that include one source file of the library and launch its kernels one by one."""
import ctypes
import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def kernel_library(tmp_path_factory, name):
    """Compile <name>_entries.cu with the library's flags, link the objects of its sources but <name>.cu."""
    import torch
    import __graft_entry__ as g
    b = g._build_module()
    objs = os.path.join(b.HERE, "_build")
    if not glob.glob(os.path.join(objs, "*.o")):
        b.build()
    out = str(tmp_path_factory.mktemp("kernels") / (name + ".so"))
    rest = [o for o in sorted(glob.glob(os.path.join(objs, "*.o"))) if os.path.basename(o) != name + ".o"]
    cmd = [b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", "-o", out, os.path.join(HERE, name + "_entries.cu"), *rest, "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(out)
