"""The beam pre-pass' launcher where the number of SMs is not known: it returns (with an error where there is no GPU, as here) and does not end the process."""
import os
import subprocess
import sys

_CALL = """
import ctypes, subprocess, sys
names = subprocess.run(["nm", "-D", "--defined-only", sys.argv[1]], check=True, capture_output=True, text=True).stdout.split()
fn = getattr(ctypes.CDLL(sys.argv[1]), next(n for n in names if "tb_launch_beam_topm" in n))
i, l, p = ctypes.c_int32, ctypes.c_int64, ctypes.c_void_p
fn.restype = ctypes.c_int
print(fn(p(0), i(1), i(2), i(3), i(2), i(20), i(20), l(126), l(42), l(21), p(0), p(0), p(0), p(0), i(15), p(0), i(int(sys.argv[2])), p(0)))
"""


def test_unknown_number_of_sms(tb):
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")            # (nothing is launched, whatever machine this is)
    codes = []
    for n_sm in ("148", "0"):
        r = subprocess.run([sys.executable, "-c", _CALL, tb.LIB_PATH, n_sm], env=env, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        codes.append(int(r.stdout))
    assert codes[0] == codes[1] < 0
