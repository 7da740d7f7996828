"""The rule that cuts a prefill call (csrc/spmm_plan.h), compiled for the host, as the library asks it on a device of 148 SMs: with the numbers of
thread-block clusters that such a device holds at once.  For tests that hold their shapes against what these are there for."""
import ctypes
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RESIDENT = [148, 148, 74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7]      # clusters of 2, 3, ... CTAs
_lib = None


def lib():
    global _lib
    if _lib is None:
        with tempfile.TemporaryDirectory() as tmp:
            out = os.path.join(tmp, "libplan_device_shim.so")
            subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                            "-o", out, os.path.join(ROOT, "tests", "plan_device_shim.cpp")], check=True)
            _lib = ctypes.CDLL(out)
        _lib.shim_device_plan.argtypes = _lib.shim_device_plan_wide.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] + [ctypes.c_void_p] * 2
        _lib.shim_pair_acc_tokens.argtypes = _lib.shim_pair_tile_tokens.argtypes = [ctypes.c_longlong]
        _lib.shim_pair_tiles_in_flight.argtypes = [ctypes.c_longlong] * 3
    return _lib


def device_plan(R, K, N, sms=148, resident=RESIDENT, wide=False):
    """wide: for 32-bit results."""
    v = (ctypes.c_longlong * 9)()
    (lib().shim_device_plan_wide if wide else lib().shim_device_plan)(R, (K + 63) // 64, N, sms, (ctypes.c_int * 17)(*resident), v)
    q = dict(zip(("kernel", "workers", "rounds", "sharers", "slices", "tiles", "rest", "cluster", "sets"), v))
    q["cut"] = q["rest"] > 0 and q["sharers"] > q["rest"]
    q["crosses"] = q["cut"] and q["kernel"] < 3 and q["sharers"] % q["rest"] > 0        # a CTA's range may end in the next tile
    return q


def pair_x_tiles(R, K, sparsity):
    """X tiles that a CTA pair has in flight."""
    return lib().shim_pair_tiles_in_flight(int(256 * R * K * (1.0 - sparsity)), R, (K + 63) // 64)
