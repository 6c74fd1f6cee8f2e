"""Device scratch of ens_mixture_host in a process of its own: the memory that its
pool keeps is bounded and goes back when a context is destroyed, a device reset
of the host program between two calls does no harm, and calls from several
threads and streams give what one call gives."""
import glob
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCRIPT = r"""
import ctypes, json, sys, threading
import numpy as np
sys.path.insert(0, sys.argv[2])
sys.path.insert(0, sys.argv[2] + "/tests")
import ens_inputs as I
from paper_2506_23712_gb300 import ens as E

rt = ctypes.CDLL(sys.argv[1])


def free():
    f, t = ctypes.c_size_t(), ctypes.c_size_t()
    assert rt.cudaMemGetInfo(ctypes.byref(f), ctypes.byref(t)) == 0
    return f.value


h = E.hist_spec(qr_bins=16, tail_bins=40)
lams = np.linspace(-1.0, 1.0, 9)
counts = I.synthetic_member_counts(lams, 16, 40, 5000, seed=1)
mom = np.random.default_rng(2).standard_normal((9, 48)) ** 2


def mix(stream=0):
    got = E.ens_mixture_host(lams, counts, mom, h, stream_ptr=stream, kind=E.W_GAUSS, mu=0.1, sigma=0.9)
    return np.concatenate([np.ravel(got[k]) for k in ("weights", "pdf_qr", "pdf_eps", "pdf_ens", "moments")])


def one_context():
    ws = None
    ms = [E.Member(N=16, nu=0.02, lam=0.0, k_lo=1, k_hi=2, dt=0.01, rk_order=2, seed=1).c()]
    ctx = ctypes.c_void_p()
    arr = (E.MemberDesc * 1)(*ms)
    assert E.lib().ens_create(arr, 1, ctypes.byref(h), None, 0, None, ctypes.byref(ctx)) == 0
    assert E.lib().ens_destroy(ctx) == 0


out = {}
ref = mix()
one_context()                     # every module loaded, nothing kept
base = free()
same = all(np.array_equal(mix(), ref) for _ in range(20))
out["kept"] = base - free()
one_context()
out["left"] = base - free()
streams = []
for _ in range(4):
    s = ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0
    streams.append(s)
bad = []


def worker(s):
    for _ in range(25):
        if not np.array_equal(mix(s), ref):
            bad.append(1)


ths = [threading.Thread(target=worker, args=(s,)) for s in streams]
[t.start() for t in ths]
[t.join() for t in ths]
out["threads"] = not bad
for _ in range(2):
    out["reset"] = rt.cudaDeviceReset()
    same = same and np.array_equal(mix(), ref) and np.array_equal(mix(), ref)
out["same"] = bool(same)
print(json.dumps(out))
"""


def test_scratch_pool():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    found = sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so.*") +
                   glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "*", "lib", "libcudart.so.*")))
    if not found:
        pytest.skip("no shared CUDA runtime to reset the device with")
    r = subprocess.run([sys.executable, "-c", SCRIPT, found[0], root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["reset"] == 0 and out["same"] and out["threads"], out
    assert 0 <= out["kept"] <= (32 << 20) + (2 << 20) and out["left"] <= 2 << 20, out
