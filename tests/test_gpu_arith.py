"""Device arithmetic of the kernels (tests/cuda/arith_probe.cu) against references of more bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1806_07390_gb300 import build as B
    so = str(tmp_path_factory.mktemp("arith") / "arith.so")
    cmd = [B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, *B.FP32_FLAGS, "-shared", "-I", B.CSRC,
           os.path.join(HERE, "cuda", "arith_probe.cu"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def on_gpu(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


# The net update of a cell in FP32: dt times the divergence, from fluxes whose directions cancel to
# 1e-6 of their parts or not at all, the lower flux far larger than the upper one among them.  The sum is
# compensated, so its error is the rounding of the result (2^-24 of it) plus second-order terms: the
# errors that are carried are below 2^-23 of the sum m of the parts' magnitudes and are themselves rounded
# a dozen times, below 2^-24 each time.
@pytest.mark.parametrize("kind", ["generic", "cancelling", "steep"])
@pytest.mark.parametrize("D", [1, 2, 3])
def test_net_update_is_compensated(probe, D, kind):
    import torch
    rng = np.random.default_rng(10 * D + len(kind))
    n = 20000
    up = rng.uniform(-1.0, 1.0, (D, n))
    lo = up * (1.0 + rng.normal(0.0, 0.05, (D, n)))
    if kind == "steep":
        lo = up * np.exp(rng.normal(0.0, 2.0, (D, n)))
    up, lo = up.astype(np.float32), lo.astype(np.float32)
    h = np.full((D, n), 0.37e-3 * 64.0, dtype=np.float32)
    if kind == "generic":
        h *= rng.uniform(0.5, 2.0, (D, 1)).astype(np.float32)
    elif D > 1:  # the last direction takes back what the others bring, to one part in a million
        net = np.sum(up[:-1].astype(np.float64) - lo[:-1], axis=0)
        lo[-1] = rng.uniform(0.1, 1.0, n).astype(np.float32)
        up[-1] = (lo[-1] - net * (1.0 + 1e-6 * rng.normal(size=n))).astype(np.float32)
    x = on_gpu(np.concatenate([np.stack([up, lo], axis=1).reshape(2 * D, n), h]))
    out = torch.zeros(2 * n, dtype=torch.float32, device="cuda")
    assert probe.arith_net(D, ptr(x), ptr(out), n) == 0
    got = out.cpu().numpy().astype(np.float64).reshape(2, n)
    u, l, f = up.astype(np.float64), lo.astype(np.float64), h.astype(np.float64)
    ref = np.sum((u - l) * f, axis=0)  # (each term exact to 2^-52 of the parts)
    m = np.sum((np.abs(u) + np.abs(l)) * f, axis=0)
    bound = 2.0 ** -24 * np.abs(ref) + 16 * 2.0 ** -47 * m + 2.0 ** -126
    assert np.array_equal(got[1], -got[0])
    assert np.all(np.abs(got[0] - ref) <= bound), np.max(np.abs(got[0] - ref) / bound)


# The channel sums of the FP32 two-equation interaction, pairs of floats: every term enters with its
# rounding error, so a sum's error is that of the low parts, each below 2^-24 of the running sum or of a
# term and rounded again twice: 2^-47 of the sum of magnitudes a term.  (A plain FP32 sum is off by 2^-25
# of the sum a term.)
def test_pair_sums_hold_twice_the_bits_of_a_float(probe):
    import torch
    rng = np.random.default_rng(5)
    n, m = 24, 4000
    x = rng.uniform(0.1, 1.0, (n, m)) * 10.0 ** rng.uniform(-3.0, 0.0, (n, m))
    y = (x * (1.0 + 1e-3 * rng.normal(size=(n, m)))).astype(np.float32)
    out = torch.zeros(3 * m, dtype=torch.float64, device="cuda")
    assert probe.arith_pairs(ptr(on_gpu(x)), ptr(on_gpu(y)), ptr(out), n, m) == 0
    got = out.cpu().numpy().reshape(3, m)
    xf, yf = x.astype(np.float32).astype(np.float64), y.astype(np.float64)
    L = np.longdouble
    for k, (terms, what) in enumerate([(xf.astype(L), "sum"), (xf.astype(L) - yf.astype(L), "difference"),
                                       (x.astype(L) * yf.astype(L), "product")]):
        size = np.sum(np.abs(xf), axis=0) if k < 2 else np.sum(np.abs(x * yf), axis=0)
        err = np.abs(got[k] - np.sum(terms, axis=0)).astype(np.float64)
        assert np.all(err <= n * 2.0 ** -47 * size), (what, np.max(err / size))
