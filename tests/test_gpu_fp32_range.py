"""fp32 storage on the tensor cores over the whole range of fp32: operands at both ends of the exponent range and operands
that are not finite, held to what fp32 FMA arithmetic gives."""
import numpy as np
import pytest
import torch

import oracle
import paper_2103_03936_b200 as pf
import pf_workloads as wl
from _gpu import dev, host

pytestmark = pytest.mark.gpu

NAMES = ("x", "U", "V", "dY")


def linear(d):
    """All results of a training step, the oracle's beside them."""
    x, U, V, dY = (dev(d[k], wl.F32) for k in NAMES)
    y, T = pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
    torch.cuda.synchronize()
    assert pf.pf_last_device_status() == 0
    got = {"y": y, "T": T, "dX": dX, "dU": dU, "dV": dV}
    with np.errstate(all="ignore"):
        want = dict(zip(("y", "T"), oracle.linear_fwd(d["x"], d["U"], d["V"])))
        want.update(zip(("dX", "dU", "dV"), oracle.linear_bwd(*(d[k] for k in NAMES))))
    return {k: host(t, wl.F32).astype(np.float64) for k, t in got.items()}, want


def conv(d, stride, pad):
    x, U, V, dY = (dev(d[k], wl.F32) for k in NAMES)
    y, T = pf.pf_lowrank_conv_fwd(x, U, V, stride=stride, pad=pad, want_stash=True)
    dX, dU, dV = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, pad=pad, T_stash=T)
    torch.cuda.synchronize()
    assert pf.pf_last_device_status() == 0
    got = {"y": y, "T": T, "dX": dX, "dU": dU, "dV": dV}
    want = dict(zip(("y", "T"), oracle.conv_fwd(d["x"], d["U"], d["V"], stride, pad)))
    want.update(zip(("dX", "dU", "dV"), oracle.conv_bwd(*(d[k] for k in NAMES), stride, pad)))
    return {k: host(t, wl.F32).astype(np.float64) for k, t in got.items()}, want


def check(got, want, tol=1e-5):
    """The same infinities and NaNs, and the finite values within `tol` (2-norm)."""
    for k in got:
        g, w = got[k], want[k]
        assert np.array_equal(np.isnan(g), np.isnan(w)), f"{k}: {np.isnan(g).sum()} NaNs, {np.isnan(w).sum()} expected"
        assert np.array_equal(np.isinf(g), np.isinf(w)) and np.array_equal(g[np.isinf(g)], w[np.isinf(w)]), f"{k}: infinities"
        f = np.isfinite(w)
        with np.errstate(all="ignore"):
            scale = np.abs(w[f]).max() if f.any() else 0.0
            err = np.linalg.norm((g[f] - w[f]) / scale) / np.linalg.norm(w[f] / scale) if scale > 0 else 0.0
        assert err <= tol, f"{k}: rel err {err:.3e}"


# sliced and whole contractions, both tile widths, operands that are copied to padded pitches (and a stash that is a second copy)
SHAPES = [(300, 520, 264, 72), (2500, 300, 1028, 40), (130, 1000, 36, 200), (257, 301, 133, 71)]


# exponents of the four operands: results stay normal fp32 numbers.  A bf16 part of an operand reaches down to 2^-133
@pytest.mark.parametrize("e", [(-124, 70, 20, 0), (-138, 70, 20, 10), (50, -125, 60, -10), (20, 10, -126, 80), (10, 20, 60, -126),
                               (118, -80, -10, 0), (-40, -40, -20, 121)], ids=str)
@pytest.mark.parametrize("m,k,n,r", SHAPES)
def test_ends_of_the_exponent_range(m, k, n, r, e):
    d = wl.LinearCase("range", m, k, n, r, wl.F32, 31).generate()
    d = {nm: np.ldexp(d[nm], s).astype(np.float32) for nm, s in zip(NAMES, e)}
    check(*linear(d))


@pytest.mark.parametrize("where", NAMES)
@pytest.mark.parametrize("m,k,n,r", SHAPES)
def test_not_finite_operands(m, k, n, r, where):
    """An infinity, a NaN and numbers within half a bf16 step of overflow reach exactly the results that FMA arithmetic
    carries them to; every other result keeps its accuracy."""
    base = wl.LinearCase("inf", m, k, n, r, wl.F32, 32).generate()
    for v in (np.inf, -np.inf, np.nan):
        d = {nm: a.copy() for nm, a in base.items()}
        d[where][7, 3] = v
        check(*linear(d))
    d = {nm: np.ldexp(a, 0 if nm == where else -10).astype(np.float32) for nm, a in base.items()}
    d[where][7, 3] = 3.3962e38
    d[where][9, 5] = -np.finfo(np.float32).max
    check(*linear(d))


def test_results_near_overflow():
    """Results up to the largest fp32 number, and sums whose terms overflow."""
    d = wl.LinearCase("big", 300, 520, 264, 72, wl.F32, 33).generate()
    d["x"] = np.ldexp(d["x"], 100).astype(np.float32)
    d["U"] = np.ldexp(d["U"], 24).astype(np.float32)      # T up to 2^127
    d["V"] = np.ldexp(d["V"], -30).astype(np.float32)
    d["dY"] = np.ldexp(d["dY"], -12).astype(np.float32)
    check(*linear(d))
    x = torch.full((300, 520), 2.0 ** 70, device="cuda")
    U = torch.full((520, 72), 2.0 ** 60, device="cuda")
    U[260:] = -2.0 ** 60
    _, T = pf.pf_lowrank_linear_fwd(x, U, torch.ones((264, 72), device="cuda"), want_stash=True)
    assert not torch.isfinite(T).any()                     # 2^130 does not exist, so neither does their sum


def test_bias_after_a_result_that_is_computed_again():
    d = wl.LinearCase("bias", 300, 520, 264, 72, wl.F32, 35).generate()
    d["x"][17, 200] = np.inf
    d["V"][100] = np.ldexp(d["V"][100], 121)               # a column whose results need the full exponent range
    b = wl.round_to(wl.normal(36, 0, (264,), 0.5), wl.F32)
    y, T = pf.pf_lowrank_linear_fwd_act(*(dev(d[k], wl.F32) for k in ("x", "U", "V")), bias=dev(b, wl.F32), want_stash=True)
    with np.errstate(all="ignore"):
        want = dict(zip(("y", "T"), oracle.linear_fwd_act(d["x"], d["U"], d["V"], b)))
    got = {"y": host(y, wl.F32).astype(np.float64), "T": host(T, wl.F32).astype(np.float64)}
    check(got, want)
    for k in ("y", "T"):                                   # and column by column, so that the large one hides none
        for c in range(0, want[k].shape[1], 25):
            check({k: got[k][:, c]}, {k: want[k][:, c]})


@pytest.mark.parametrize("N,H,W,C,R,O,k,stride,pad,at", [
    (2, 13, 6, 36, 20, 24, 3, 1, 0, (0, 11, 2, 5)),       # the last block of pixels reaches past the last output row
    (2, 9, 43, 36, 20, 24, 3, 1, 0, (1, 4, 41, 5)),       # ... past the last output column
    (3, 11, 13, 100, 12, 40, 3, 2, 1, (2, 4, 6, 99)),
    (5, 5, 5, 64, 16, 64, 3, 1, 1, (4, 0, 0, 63)),
    (6, 56, 56, 132, 72, 40, 3, 1, 1, (5, 30, 31, 131))])      # tiles of 128 columns
def test_convolution_range(N, H, W, C, R, O, k, stride, pad, at):
    """The convolution's products on the same kernel: an infinite input or gradient reaches its own window only, small and
    large operands keep fp32 accuracy."""
    base = wl.ConvCase("crange", N, H, W, C, R, O, wl.F32, 34, kh=k, kw=k, stride=stride, pad=pad).generate()
    for nm, v in (("x", np.inf), ("x", np.nan), ("dY", -np.inf)):
        d = {n2: a.copy() for n2, a in base.items()}
        if nm == "x":
            d[nm][at] = v
        else:
            d[nm][at[0], d[nm].shape[1] // 2, d[nm].shape[2] // 2, 3] = v     # (its window holds no padding: 0 * inf is NaN)
        check(*conv(d, stride, pad))
    for e in ((-130, 60, 20, 10), (118, -60, -20, 0)):
        d = {nm: np.ldexp(base[nm], s).astype(np.float32) for nm, s in zip(NAMES, e)}
        check(*conv(d, stride, pad))


def test_long_contraction_of_one_sign():
    """dV over 65536 equal rows (slices of 32768): every operand is 1 + just under 2^-8, so that a1 b1 = 1 sums exactly and
    all of the error is that of the correction products, of one sign and as large as they can be.  Their
    accumulator takes 2048 elements: 640 additions, each truncated by at most an ulp, 2^-23 of at most 2^-7 of the sum of
    those elements: 6.0e-7 of the result.  The 16 drains of a slice and 9 doublings of its sum round it by at most 2^-24 of what it is
    then, half of the end's on average, and with equal addends in one direction: 25 * 2^-25 = 7.5e-7.  (One accumulator for
    the whole slice: 6.9e-6.)"""
    m, n, r, k = 65536, 1024, 512, 32
    a = 1 + 2.0 ** -8 * np.random.default_rng(1).uniform(0.9, 0.999, n)
    b = 1 + 2.0 ** -8 * np.random.default_rng(2).uniform(0.9, 0.999, r)
    a, b = a.astype(np.float32), b.astype(np.float32)
    dY = torch.from_numpy(a).cuda().expand(m, n).contiguous()
    T = torch.from_numpy(b).cuda().expand(m, r).contiguous()
    x, U, V = torch.ones((m, k), device="cuda"), torch.ones((k, r), device="cuda"), torch.ones((n, r), device="cuda")
    _, _, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T, need_dX=False)
    want = m * np.outer(a.astype(np.float64), b.astype(np.float64))
    rel = np.abs(host(dV, wl.F32).astype(np.float64) - want) / want
    assert rel.max() <= 1.35e-6, f"{rel.max():.3e}"
