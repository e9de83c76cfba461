"""A launch that fails is reported by the call that made it, with the error's name, and
leaves nothing for a later call to find (no GPU: every launch fails)."""
import subprocess
import sys

import pytest


def test_every_call_names_its_cuda_error():
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("launches succeed here")
    from paper_2405_18628_gb300 import build, ppd
    build.build()
    # a process's first failure names its error, so each call gets a process of its own
    code = ("import ctypes, sys; from paper_2405_18628_gb300 import ppd; lib = ppd.load(); f = ctypes.c_void_p(0x10000); "
            "st = {}; print(st, lib.ppd_last_cuda_error().decode())")
    for call in ("lib.ppd_node_argmax_noalloc(f, 1, 4, 16, f, None)",
                 "lib.ppd_node_argmax(f, 1, 4, 16, f, f, 1 << 30, None)",
                 "lib.ppd_accept_path(f, f, f, f, 1, 4, 16, 8, f, f, f, f, f, None)",
                 "lib.ppd_kv_compact(f, ctypes.c_void_p(0x100000), ctypes.c_void_p(0x200000), ctypes.c_void_p(0x300000), "
                 "f, f, f, 1, 1, 1, 4, 64, 8, 0, None)",
                 "lib.ppd_next_tree(*[f] * 6, 2, 16, 100, 4, 32, f, f, 4, 1, *[f] * 4, f, 1 << 20, None)"):
        r = subprocess.run([sys.executable, "-c", code.format(call)], capture_output=True, text=True, check=True)
        status, name = r.stdout.split()
        assert int(status) == ppd.PPD_ERR_CUDA, (call, r.stdout)
        assert name.startswith("cudaError"), (call, name)
