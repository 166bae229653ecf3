"""Device arithmetic of the kernels (tests/cuda/arith_probe.cu) against references of more bits."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1806_07390_gb300 import fx
from paper_1806_07390_gb300 import workloads as W

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


FP64 = ["rcp64", "rcp_pos", "rcp_any", "rcp_fast", "rcp_ge1", "sqrt64", "sqrt_any", "rsqrt64"]
U = 2.0 ** -53


def fp64(probe, name, x):
    import torch
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = torch.zeros(x.size, dtype=torch.float64, device="cuda")
    assert probe.arith_fp64(FP64.index(name), ptr(on_gpu(x)), ptr(out), x.size) == 0
    return out.cpu().numpy()


def spread(lo, hi, n, seed):
    """Numbers over the binades lo .. hi - 1 with random mantissas, and each binade's ends."""
    rng = np.random.default_rng(seed)
    e = rng.integers(lo, hi, n)
    ends = np.ldexp(1.0, np.arange(lo, hi))
    return np.concatenate([np.ldexp(rng.uniform(1.0, 2.0, n), e), ends, np.nextafter(2.0 * ends, 0.0)])


# The short FP64 reciprocals and roots over their stated domains.  A reciprocal's last operation is one FMA,
# half a unit (U relative), on a correction whose own error is e^3 < 2^-57 = U/16; the square root ends
# on the rounded correction of a value good to 2^-38, whose square is far below U; the reciprocal root adds to
# its own half unit that of a y (half a unit of y^2 a, halved by the series).
@pytest.mark.parametrize("name,lo,hi,bound", [
    ("rcp64", -1022, 1022, 1.07), ("rcp_pos", -1022, 1022, 1.07), ("rcp_fast", -1022, 1022, 1.07),
    ("rcp_any", -1021, 1022, 1.07), ("rcp_ge1", 0, 1021, 1.07), ("sqrt64", -1021, 1020, 1.02),
    ("sqrt_any", -1021, 1023, 1.02), ("rsqrt64", -1021, 1020, 1.6)])
def test_fp64_reciprocals_and_roots(probe, name, lo, hi, bound):
    x = spread(lo, hi, 100000, 7)
    got, L = fp64(probe, name, x).astype(np.longdouble), x.astype(np.longdouble)
    ref = np.sqrt(L) if "sqrt" in name and name[0] == "s" else 1 / (np.sqrt(L) if name == "rsqrt64" else L)
    err = np.abs(got / ref - 1).astype(np.float64)
    assert np.max(err) <= bound * U, (np.max(err) / U, x[np.argmax(err)])


def test_fp64_reciprocals_and_roots_at_the_ends(probe):
    inf, nan, tiny = np.inf, np.nan, 5e-324
    edge = [0.0, inf, nan, tiny, 2.0 ** -1022, 2.0 ** 1022, 2.0 ** 1023, np.finfo(float).max]
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / np.array(edge)
    got = fp64(probe, "rcp_any", edge + [-e for e in edge])
    np.testing.assert_array_equal(got, np.concatenate([want, -want]))
    np.testing.assert_array_equal(fp64(probe, "rcp_pos", [1.0, inf]), [1.0, 0.0])
    # past 2^1022 the closure's factor and the optical depth's are 0 or denormal, at infinity 0
    assert np.all(np.abs(fp64(probe, "rcp_fast", [2.0 ** 1023, np.finfo(float).max, inf])) <= 2.0 ** -1022)
    np.testing.assert_array_equal(fp64(probe, "rcp_ge1", [0.0, 0.5, 1.0, 2.0, 2.0 ** 1022, inf]), [1, 1, 1, 0.5, 0, 0])
    np.testing.assert_array_equal(fp64(probe, "sqrt_any", [0.0, inf, nan, -1.0, tiny, 4.0]),
                                  [0.0, inf, nan, nan, np.sqrt(tiny), 2.0])
    assert np.isnan(fp64(probe, "rcp64", [nan])[0]) and np.isnan(fp64(probe, "rcp_fast", [nan])[0])


# x^(h/2): one rounding per product (n of them for the power k = floor(h/2), and one for the root), the
# reciprocal's and the root's own
def test_fp64_half_integer_powers(probe):
    import torch
    rng = np.random.default_rng(3)
    h = np.repeat(np.arange(-14, 15), 2000).astype(np.int32)
    x = 10.0 ** rng.uniform(-8.0, 8.0, h.size)
    out = torch.zeros(h.size, dtype=torch.float64, device="cuda")
    assert probe.arith_hpow(ptr(on_gpu(x)), ptr(on_gpu(h)), ptr(out), h.size) == 0
    L = x.astype(np.longdouble)
    k = h >> 1
    ref = np.ones_like(L)
    for _ in range(7):
        ref = np.where(np.abs(k) > _, ref * L, ref)
    ref = np.where(k < 0, 1 / ref, ref) * np.where(h & 1, np.sqrt(L), 1)
    err = np.abs(out.cpu().numpy().astype(np.longdouble) / ref - 1).astype(np.float64)
    bound = (np.maximum(np.abs(k) - 1, 0) + np.where(k < 0, 1.07, 0.0) + np.where(h & 1, 2.02, 0.0)) * U
    assert np.all(err <= 1.001 * bound), np.max(err / np.maximum(bound, U))


def planck_reference(x):
    """(lower integral, upper integral, w) in long double: the power series in the Bernoulli numbers below 3.2,
    the exponential series above 2.8 (each to 1e-25 of its value there; NaN elsewhere)."""
    L = np.longdouble
    b, fact = [Fraction(1)], [Fraction(1)]
    for k in range(1, 90):
        fact.append(fact[-1] * k)
    for k in range(1, 89):
        b.append(-sum(b[j] / fact[k + 1 - j] for j in range(k)))
    f = [L(v.numerator) / L(v.denominator) if abs(v.denominator) < 10 ** 4000 else L(0) for v in b]
    x = x.astype(L)
    lo = np.full(x.shape, L(np.nan))
    s = x < 3.2
    t = np.zeros(int(s.sum()), dtype=L)
    for m in range(44, 0, -1):
        t = t * x[s] ** 2 + f[2 * m] / (2 * m + 3)
    lo[s] = x[s] ** 3 * (L(1) / 3 - x[s] / 8 + t * x[s] ** 2)
    up = np.full(x.shape, L(np.nan))
    s = x > 2.8
    v, t = x[s], np.zeros(int(s.sum()), dtype=L)
    for n in range(1, 25):
        t += np.exp(-n * v) * (v ** 3 / n + 3 * v ** 2 / L(n) ** 2 + 6 * v / L(n) ** 3 + 6 / L(n) ** 4)
    up[s] = t
    return lo, up, x ** 4 / np.expm1(x)


# The band edges from the table of polynomials, on both sides of the rows where the integral changes ends and
# where the table ends.  A polynomial's value takes two units of 2^-53 (its leading coefficient's rounding
# and the last FMA's; the others enter with t^k, |t| <= 1/2, and small ratios), its derivative three.  The
# integral: x^3 and the product with it, three more.  Its weight: two for x^3, one each for 3 p, the FMA and
# the product, on three.  Past the table the exponential series, whose exponential, sum and quotient take
# eight.
def test_planck_edges_from_the_table(probe):
    import torch
    rng = np.random.default_rng(11)
    x16 = np.concatenate([rng.uniform(0.0, 1024.0, 20000), 10.0 ** rng.uniform(-4.0, 1.0, 4000), np.arange(1.0, 1025.0),
                          np.arange(1.0, 1024.0) + 0.5, rng.uniform(47.0, 48.0, 4000), rng.uniform(1023.0, 1025.0, 2000),
                          rng.uniform(1024.0, 8000.0, 2000)])
    n = x16.size
    out = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    assert probe.arith_planck_edge(ptr(on_gpu(x16)), ptr(out), n) == 0
    Q, w, upper = out.cpu().numpy().reshape(3, n)
    np.testing.assert_array_equal(upper, np.rint(x16) >= 48)
    lo, up, wr = planck_reference(x16 / 16.0)
    ref = np.where(upper == 1.0, up, lo)
    assert np.all(np.isfinite(ref))
    eq, ew = np.abs(Q / ref - 1).astype(np.float64) / U, np.abs(w / wr - 1).astype(np.float64) / U
    tab = x16 < 1024.0
    assert np.max(eq[tab]) <= 5.0 and np.max(ew[tab]) <= 8.0, (np.max(eq[tab]), np.max(ew[tab]))
    assert np.max(eq[~tab]) <= 8.0 and np.max(ew[~tab]) <= 8.0, (np.max(eq[~tab]), np.max(ew[~tab]))


# The FP32 band table as the device holds it (two groups' coefficients interleaved, the scale's exponent in
# the low bits of the last one), in both layouts, for odd and even group counts and one group, against the
# oracle.  T sits at u = log2 T with an error of 2 units of log2f and one of the difference to the table's
# start (2e-6 together), and d ln I / d ln T is at most x + 4, x = eps/T at the lower edge; the interpolation
# and its evaluation add 1e-6.
@pytest.mark.parametrize("node_major", [0, 1])
@pytest.mark.parametrize("G", [1, 2, 7, 16])
def test_planck_bands_from_the_device_table(probe, G, node_major):
    import torch

    import oracle
    pb, _ = W.kh_2d(nx=16, ny=16, ngroups=G)
    P, h, ws = fx.params(pb), ctypes.c_void_p(), ctypes.c_size_t()
    L = fx.lib()
    assert L.fx_grid_create(ctypes.byref(P), ctypes.byref(h), ctypes.byref(ws)) == 0
    nu, u0 = ctypes.c_int(), ctypes.c_float()
    size = L.fx_debug_planck_table(h, None, 0, ctypes.byref(nu), ctypes.byref(u0))
    nodes = np.zeros(size, dtype=np.float32)
    fp = ctypes.POINTER(ctypes.c_float)
    L.fx_debug_planck_table(h, nodes.ctypes.data_as(fp), size, ctypes.byref(nu), ctypes.byref(u0))
    L.fx_grid_destroy(h)
    edges = pb.eps_min * (pb.eps_max / pb.eps_min) ** (np.arange(G + 1) / G)
    e32 = edges.astype(np.float32)
    rng = np.random.default_rng(G)
    # random temperatures over the table's useful range, and every node of two octaves from both sides
    node = 2.0 ** (-1.0 + np.arange(65) / 32.0)
    T = np.concatenate([np.exp(rng.uniform(np.log(0.02), np.log(200.0), 400)), node * (1 - 1e-5), node * (1 + 1e-5)])
    T = T.astype(np.float32)
    n = T.size
    out = torch.zeros(2 * G * n, dtype=torch.float32, device="cuda")
    f = ctypes.c_float
    assert probe.arith_planck_bands(nodes.ctypes.data_as(fp), G, nu.value, f(u0.value), node_major, e32.ctypes.data_as(fp),
                                    ptr(on_gpu(T)), ptr(out), n) == 0
    B, dB = out.cpu().numpy().astype(np.float64).reshape(2, G, n)
    aN = pb.a_rad * 15.0 / np.pi ** 4
    checked = 0
    for i, t in enumerate(T.astype(np.float64)):
        for g in range(G):
            rb, rd = oracle.planck_group(pb, g, t)
            rb, rd = rb / aN, rd / aN
            # (the FP32 units flush denormals: the band's 2^k, and B and B/T themselves)
            if rb / t ** 4 < 2.0 ** -120 or min(rb, rb / t) < 2.0 ** -125:
                continue
            x = edges[g] / t
            assert abs(B[g, i] - rb) <= (2e-6 * (x + 4.0) + 1e-6) * rb, (g, t, B[g, i], rb)
            # dB/dT = T^3 I (4 + d): the bound of I, and that of d on the scale of one
            assert abs(dB[g, i] - rd) <= (2e-6 * (x + 4.0) + 1e-6) * (abs(rd) + (x + 4.0) * rb / t), (g, t, dB[g, i], rd)
            checked += 1
    assert checked > 0.5 * n * G
