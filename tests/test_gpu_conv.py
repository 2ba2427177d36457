"""GPU parity: factorized NHWC convolution forward/backward through the C ABI vs the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2103_03936_b200 as pf
import pf_workloads as wl
from _gpu import ESCAPES, PFDT, Guarded, Scratch, assert_blocks_close, assert_close, dev

pytestmark = pytest.mark.gpu


def run_conv(case, stash=True, need_dX=True, tiny=False, bwd_room=None):
    d = case.generate()
    dt = case.dtype
    x, U, V, dY = (dev(d[k_], dt) for k_ in ("x", "U", "V", "dY"))
    Ho, Wo = case.Ho, case.Wo
    gy = Guarded((case.N, Ho, Wo, case.O), dt)
    gT = Guarded((case.N, Ho, Wo, case.R), dt)
    scratch = [Scratch(pf.pf_lowrank_conv_workspace(case.N, case.H, case.W, case.C, case.R, case.O, case.kh, case.kw, case.stride, case.pad, PFDT[dt], bwd)
                       if not (bwd and bwd_room) else bwd_room) for bwd in (False, True)]
    pf.pf_lowrank_conv_fwd(x, U, V, stride=case.stride, pad=case.pad, y=gy.t,
                           T_stash=gT.t if stash else None, workspace=scratch[0].t)
    gdX, gdU, gdV = Guarded(x.shape, dt), Guarded(U.shape, dt), Guarded(V.shape, dt)
    pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=case.stride, pad=case.pad,
                           T_stash=gT.t if stash else None, need_dX=need_dX,
                           dX=gdX.t if need_dX else None, dU=gdU.t, dV=gdV.t, workspace=scratch[1].t)
    torch.cuda.synchronize()
    y_ref, T_ref = oracle.conv_fwd(d["x"], d["U"], d["V"], case.stride, case.pad)
    dX_ref, dU_ref, dV_ref = oracle.conv_bwd(d["x"], d["U"], d["V"], d["dY"], case.stride, case.pad)
    ab = {}
    if tiny:   # magnitude of the summands, for outputs of a handful of elements
        aw = {k_: np.abs(oracle.widen(v)) for k_, v in d.items()}
        ab["y"], ab["T"] = oracle.conv_fwd(aw["x"], aw["U"], aw["V"], case.stride, case.pad)
        ab["dX"], ab["dU"], ab["dV"] = oracle.conv_bwd(aw["x"], aw["U"], aw["V"], aw["dY"], case.stride, case.pad)
    tag = f"{case.name} {case.N}x{case.H}x{case.W} {case.C}->{case.R}->{case.O} k{case.kh} s{case.stride} {dt} "
    checks = [("y", gy, y_ref)]
    if stash:
        checks.append(("T", gT, T_ref))
    if need_dX:
        checks.append(("dX", gdX, dX_ref))
    checks += [("dU", gdU, dU_ref), ("dV", gdV, dV_ref)]
    errs = {nm: assert_close(g.t, ref, dt, tag + nm, abs_ref64=ab.get(nm)) for nm, g, ref in checks}
    for g in (gy, gT, gdX, gdU, gdV, *scratch):
        g.check()
    assert pf.pf_last_device_status() == 0
    return errs


SMALL = [  # N,H,W,C,R,O,k,stride,pad
    (1, 1, 1, 1, 1, 1, 1, 1, 0),
    (1, 3, 3, 1, 1, 1, 3, 1, 1),
    (2, 5, 4, 3, 2, 3, 3, 1, 1),
    (1, 6, 5, 2, 3, 2, 3, 2, 1),
    (2, 4, 4, 2, 2, 3, 1, 1, 0),
    (1, 5, 5, 2, 2, 2, 3, 1, 0),
    (1, 7, 6, 2, 2, 2, 5, 2, 2),
    (3, 9, 11, 8, 5, 16, 3, 1, 1),
    (2, 8, 8, 16, 8, 24, 3, 1, 1),
]


# bf16 outputs of the small shapes that may be measured against the magnitude of their summands
# (single near-cancelled sums, see _gpu.assert_close); fixed by the seeded inputs.
MAX_CANCELLED_OUTPUTS = 1


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_small_shapes(dtype):
    first = len(ESCAPES)
    for i, (N, H, W, C, R, O, k, st, pad) in enumerate(SMALL):
        run_conv(wl.ConvCase(f"s{i}", N, H, W, C, R, O, dtype, 50 + i, kh=k, kw=k, stride=st, pad=pad), tiny=True)
    took = ESCAPES[first:]
    for what, rel, ratio, err_abs in took:
        print(f"cancelled output {what}: rel {rel:.2e}, |exact|/|summands| {ratio:.2e}, err vs summands {err_abs:.2e}")
    assert len(took) <= (MAX_CANCELLED_OUTPUTS if dtype == wl.BF16 else 0), took


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
@pytest.mark.parametrize("N,H,W,C,R,O", [(2, 32, 32, 64, 16, 64), (3, 14, 14, 64, 16, 128),
                                         (1, 20, 12, 72, 24, 40), (5, 16, 16, 128, 32, 128)])
def test_multi_tile(dtype, N, H, W, C, R, O):
    run_conv(wl.ConvCase("mt", N, H, W, C, R, O, dtype, 60))


@pytest.mark.parametrize("N,H,W,C,R,O,k", [(2, 32, 32, 128, 64, 128, 3), (3, 16, 16, 256, 64, 64, 3),
                                           (2, 16, 32, 128, 64, 96, 3), (1, 64, 64, 128, 64, 128, 3),
                                           (2, 32, 32, 128, 128, 256, 5), (2, 8, 16, 128, 192, 64, 1),
                                           (3, 14, 14, 128, 64, 128, 3), (2, 7, 7, 256, 64, 64, 3),
                                           (2, 28, 28, 128, 64, 72, 3), (3, 10, 6, 128, 64, 64, 3),
                                           (1, 3, 64, 128, 64, 64, 3),
                                           (2, 16, 16, 128, 256, 64, 3), (2, 16, 16, 128, 320, 128, 3),
                                           (2, 16, 16, 128, 384, 72, 3)])
def test_tensor_core_envelope(N, H, W, C, R, O, k):
    """Stride-1, 'same'-padded shapes whose channels fill the 64-channel blocks of the implicit GEMMs and whose image rows
    pack into 128- and 64-pixel tiles (other tilings: below), with and without stash / dX.  The
    ranks 256, 320 and 384 reach the parts of the fused kernel that only ranks above 192 use (a
    second group of first-product MMAs, the short ring, store staging inside the ring stages)."""
    run_conv(wl.ConvCase("tc", N, H, W, C, R, O, wl.BF16, 63, kh=k, kw=k, pad=(k - 1) // 2))
    run_conv(wl.ConvCase("tc", N, H, W, C, R, O, wl.BF16, 64, kh=k, kw=k, pad=(k - 1) // 2), stash=False,
             need_dX=False)


def test_recompute_without_stash_and_no_dX():
    run_conv(wl.ConvCase("ns", 2, 16, 16, 64, 16, 64, wl.BF16, 61), stash=False)
    run_conv(wl.ConvCase("nx", 2, 16, 16, 64, 16, 64, wl.BF16, 62), need_dX=False)


@pytest.mark.parametrize("name,imgs", [("C4", [0, 63, 127]), ("C5b", [0, 100, 255])])
def test_configs_full_size_sampled(name, imgs):
    """Full-size conv configs: y, T, dX on sampled images (exact per image), dU, dV on sampled
    rank columns (exact from column-sliced factors)."""
    c = wl.conv_cases()[name]
    d = c.generate()
    x, U, V, dY = (dev(d[k_], c.dtype) for k_ in ("x", "U", "V", "dY"))
    y, T = pf.pf_lowrank_conv_fwd(x, U, V, want_stash=True)
    dX, dU, dV = pf.pf_lowrank_conv_bwd(x, U, V, dY, T_stash=T)
    torch.cuda.synchronize()
    y_ref, T_ref = oracle.conv_fwd(d["x"][imgs], d["U"], d["V"])
    dX_ref, _, _ = oracle.conv_bwd(d["x"][imgs], d["U"], d["V"], d["dY"][imgs])
    for got, want, nm in ((y[imgs], y_ref, "y"), (T[imgs], T_ref, "T"), (dX[imgs], dX_ref, "dX")):
        assert_close(got, want, c.dtype, nm)
        assert_blocks_close(got, want, c.dtype, nm)          # 128 pixels x 128 channels per block
    J = [0, 31, 63]
    _, dU_ref, dV_ref = oracle.conv_bwd(d["x"], d["U"][..., J], d["V"][:, J], d["dY"])
    for got, want, nm in ((dU[..., J], dU_ref, "dU"), (dV[:, J], dV_ref, "dV")):
        assert_close(got, want, c.dtype, nm)
        assert_blocks_close(got, want, c.dtype, nm)          # 128 rows x the sampled columns per block
    # the step ends with the flat gradient buffer of its factor gradients
    flat, offs = pf.pf_pack_factor_grads([dU, dV])
    torch.cuda.synchronize()
    assert offs == [0, dU.numel(), dU.numel() + dV.numel()]
    assert torch.equal(flat[:offs[1]], dU.reshape(-1)) and torch.equal(flat[offs[1]:], dV.reshape(-1))
    assert pf.pf_last_device_status() == 0


def test_backward_is_bit_reproducible():
    """dU and dV are sums over all pixels split across CTAs; the slices are added in a fixed order."""
    c = wl.ConvCase("rep", 8, 32, 32, 128, 64, 128, wl.BF16, 31)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V", "dY"))
    a = pf.pf_lowrank_conv_bwd(x, U, V, dY)
    b = pf.pf_lowrank_conv_bwd(x, U, V, dY)
    torch.cuda.synchronize()
    for p, q in zip(a, b):
        assert torch.equal(p, q)
    assert pf.pf_last_device_status() == 0


def test_empty_batch():
    x = torch.empty((0, 8, 8, 8), dtype=torch.bfloat16, device="cuda")
    U = torch.ones((3, 3, 8, 4), dtype=torch.bfloat16, device="cuda")
    V = torch.ones((8, 4), dtype=torch.bfloat16, device="cuda")
    y = pf.pf_lowrank_conv_fwd(x, U, V)
    assert y.shape == (0, 8, 8, 8)
    _, dU, dV = pf.pf_lowrank_conv_bwd(x, U, V, torch.empty((0, 8, 8, 8), dtype=torch.bfloat16, device="cuda"))
    torch.cuda.synchronize()
    assert torch.all(dU == 0) and torch.all(dV == 0)


@pytest.mark.parametrize("dtype,N,H,W,C,R,O,stride", [(wl.BF16, 4, 16, 16, 128, 64, 128, 1), (wl.BF16, 2, 8, 8, 24, 8, 16, 2),
                                                      (wl.BF16, 2, 8, 8, 20, 6, 12, 2), (wl.F32, 2, 8, 8, 16, 8, 24, 1)])
def test_conv_grads_fp32_and_accumulated(dtype, N, H, W, C, R, O, stride):
    """pf_lowrank_conv_bwd_ex: fp32 factor gradients reproduce the plain call when rounded (same sums),
    and accumulation over two halves of the batch gives the whole batch's gradient on top of the
    previous contents; tensor cores at both strides, FMA kernels (channels that are no multiples of 8), fp32 storage."""
    c = wl.ConvCase("cg", N, H, W, C, R, O, dtype, 71, stride=stride)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], dtype) for k_ in ("x", "U", "V", "dY"))
    _, dU0, dV0 = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, need_dX=False)
    _, dU1, dV1 = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, need_dX=False, grads_f32=True)
    assert dU1.dtype == torch.float32 and torch.equal(dU1.to(dU0.dtype), dU0) and torch.equal(dV1.to(dV0.dtype), dV0)
    _, dU_ref, dV_ref = oracle.conv_bwd(d["x"], d["U"], d["V"], d["dY"], stride=stride, pad=1)
    tol = 1e-2 if dtype == wl.BF16 else 1e-4
    assert_close(dU1, dU_ref, wl.F32, "conv fp32 dU", tol=tol)
    assert_close(dV1, dV_ref, wl.F32, "conv fp32 dV", tol=tol)
    prevU = torch.full(U.shape, 0.25, dtype=torch.float32, device="cuda")
    prevV = torch.full(V.shape, -0.5, dtype=torch.float32, device="cuda")
    h = N // 2
    for lo, hi in ((0, h), (h, N)):
        pf.pf_lowrank_conv_bwd(x[lo:hi], U, V, dY[lo:hi], stride=stride, need_dX=False, dU=prevU, dV=prevV,
                               accumulate=True, grads_f32=True)
    torch.cuda.synchronize()
    assert_close(prevU, 0.25 + dU_ref, wl.F32, "conv accumulated dU", tol=tol)
    assert_close(prevV, -0.5 + dV_ref, wl.F32, "conv accumulated dV", tol=tol)
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("N,H,W,C,R,O", [(4, 16, 16, 128, 64, 128), (3, 14, 14, 256, 64, 256), (2, 15, 17, 128, 128, 72),
                                         (40, 32, 32, 128, 64, 256)])
def test_stride2_forward_on_tensor_cores(N, H, W, C, R, O):
    """Stride-2 3 x 3 convolutions (the first convolution of a ResNet stage): the forward runs on the fused
    tensor-core kernel with image tiles fetched two pixels apart (one launch; even and odd image sizes,
    output rows that do not fill a tile, more tiles than SMs), and the backward on the tensor cores too."""
    c = wl.ConvCase("s2", N, H, W, C, R, O, wl.BF16, 81, stride=2)
    d = c.generate()
    x, U, V = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V"))
    gy = Guarded((N, c.Ho, c.Wo, O), wl.BF16)
    gT = Guarded((N, c.Ho, c.Wo, R), wl.BF16)
    l0 = pf.pf_launch_count()
    pf.pf_lowrank_conv_fwd(x, U, V, stride=2, pad=1, y=gy.t, T_stash=gT.t)
    assert pf.pf_launch_count() - l0 == 1
    torch.cuda.synchronize()
    y_ref, T_ref = oracle.conv_fwd(d["x"], d["U"], d["V"], 2, 1)
    assert_close(gy.t, y_ref, wl.BF16, "stride-2 y")
    assert_close(gT.t, T_ref, wl.BF16, "stride-2 T")
    assert_blocks_close(gy.t, y_ref, wl.BF16, "stride-2 y", br=32)
    gy.check()
    gT.check()
    assert pf.pf_last_device_status() == 0
    run_conv(c)          # and the whole forward + backward against the oracle


@pytest.mark.parametrize("N,H,W,C,R,O,k,stride,pad", [
    (5, 5, 5, 64, 16, 64, 3, 1, 1),      # several whole images per tile (a ragged last group), one 64-channel block per tap
    (3, 7, 7, 96, 24, 40, 3, 1, 1),      # ragged channel block, 49-pixel reduction blocks (zero-filled tail)
    (2, 13, 11, 72, 8, 16, 3, 1, 1),     # image rows that do not divide into tiles
    (4, 9, 9, 160, 40, 80, 3, 2, 1),     # stride 2, odd image: four pixel classes of unequal size
    (7, 4, 6, 128, 80, 256, 3, 2, 1),    # stride 2, several images per tile, ranks past one 64-block
    (2, 12, 12, 64, 16, 72, 5, 3, 2),    # stride 3, 5 x 5 taps
    (3, 6, 6, 32, 16, 24, 3, 1, 0),      # no padding: fewer output than input pixels
    (2, 16, 16, 24, 8, 16, 2, 2, 0),     # one tap per class
    (150, 4, 4, 64, 16, 64, 3, 1, 1),
])
def test_tensor_core_tilings(N, H, W, C, R, O, k, stride, pad):
    """Edges of the implicit-GEMM tilings: tiles of several images, rows that do not divide, ragged channel
    blocks and strided backward passes, with and without stash / dX; fp32 gradients from the slices."""
    c = wl.ConvCase("til", N, H, W, C, R, O, wl.BF16, 91, kh=k, kw=k, stride=stride, pad=pad)
    run_conv(c)
    run_conv(c, stash=False, need_dX=False)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V", "dY"))
    _, dU0, dV0 = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, pad=pad)
    _, dU1, dV1 = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, pad=pad, grads_f32=True)
    torch.cuda.synchronize()
    assert torch.equal(dU1.to(dU0.dtype), dU0) and torch.equal(dV1.to(dV0.dtype), dV0)


@pytest.mark.parametrize("N,H,W,C,R,O,k,stride,pad", [(2, 9, 40, 36, 20, 24, 3, 1, 1), (5, 5, 5, 64, 16, 64, 3, 1, 1), (3, 11, 13, 100, 12, 40, 3, 2, 1),
                                                      (1, 6, 6, 32, 132, 64, 3, 1, 0), (2, 12, 12, 64, 32, 72, 5, 3, 2),
                                                      (2, 300, 3, 8, 8, 12, 3, 3, 1), (1, 520, 4, 12, 4, 8, 4, 4, 0)])
def test_fp32_tensor_core_tilings(N, H, W, C, R, O, k, stride, pad):
    """fp32 convolutions through the split-operand kernel: image rows longer than a reduction block, several images per
    tile, ragged channel blocks, strided backward, strided images one output pixel wide (boxes of input rows are at most
    256 high); held to fp32 accuracy."""
    errs = run_conv(wl.ConvCase("f32tc", N, H, W, C, R, O, wl.F32, 93, kh=k, kw=k, stride=stride, pad=pad))
    assert max(errs.values()) <= 1e-5, errs
    run_conv(wl.ConvCase("f32tc", N, H, W, C, R, O, wl.F32, 94, kh=k, kw=k, stride=stride, pad=pad), stash=False, need_dX=False)


@pytest.mark.parametrize("N,H,W,C,R,O", [(170, 15, 17, 64, 16, 72), (600, 7, 9, 72, 24, 40), (3000, 4, 4, 64, 64, 136), (12, 56, 56, 128, 40, 64), (1300, 6, 5, 64, 64, 256)])
def test_resident_image_windows(N, H, W, C, R, O):
    """Many tiles of a 3 x 3, stride-1 convolution: the flat image sequence (a zero column and row between images) whose
    windows serve all taps; tiles across image borders, boxes of rows and of whole images, ragged channel blocks."""
    run_conv(wl.ConvCase("res", N, H, W, C, R, O, wl.BF16, 95))


@pytest.mark.parametrize("N,H,W,C,R,O", [
    (45, 16, 16, 320, 40, 72),       # 16 divides the width: dU's blocks take the image's columns; an odd number of channel blocks; half a tile of dY
    (8, 32, 48, 264, 56, 136),       # blocks of one row of 48; a ragged channel block
    (300, 7, 7, 256, 40, 64),        # blocks of whole images
    (140, 9, 13, 136, 24, 136),      # rows that do not divide into blocks
    (13, 33, 63, 72, 24, 72),        # the widest image; one block of channels, ragged
    (950, 3, 4, 512, 40, 24),        # windows of dX in boxes of whole images
    (16, 32, 32, 512, 40, 512),      # the widest y
    (60, 31, 15, 192, 48, 96),
    (60, 28, 28, 128, 8, 128),       # one block of channels, the smallest rank
])
def test_flat_backward(N, H, W, C, R, O):
    """3 x 3, stride-1 backwards in three launches that read their images once: edges of their blocks, with and without
    stash and dX; gradients in fp32 are the sums that the plain ones are rounded from."""
    c = wl.ConvCase("flat", N, H, W, C, R, O, wl.BF16, 97)
    run_conv(c)
    run_conv(c, stash=False, need_dX=False)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V", "dY"))
    before = pf.pf_launch_count()
    _, dU0, dV0 = pf.pf_lowrank_conv_bwd(x, U, V, dY)
    assert pf.pf_launch_count() - before == (5 if N * H * W >= 20000 and R % 16 and 64 % R else 4)         # (x U once more; many pixels: U copied where its rows straddle lines)
    _, dU1, dV1 = pf.pf_lowrank_conv_bwd(x, U, V, dY, grads_f32=True)
    torch.cuda.synchronize()
    assert torch.equal(dU1.to(dU0.dtype), dU0) and torch.equal(dV1.to(dV0.dtype), dV0)


@pytest.mark.parametrize("N,H,W,C,R,O", [(80, 16, 16, 320, 40, 72), (70, 28, 28, 72, 24, 72), (27, 33, 63, 264, 8, 72)])
def test_flat_backward_into_the_callers_sums(N, H, W, C, R, O):
    """Gradients in fp32 or accumulated come from the launches of the plain ones, wherever the matrices lie: the fp32 sums that
    the plain ones are rounded from, added once to what was there."""
    c = wl.ConvCase("sums", N, H, W, C, R, O, wl.BF16, 94)
    run_conv(c, need_dX=False)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V", "dY"))
    T = pf.pf_lowrank_conv_fwd(x, U, V, want_stash=True)[1]
    for dX in (True, False):
        before = pf.pf_launch_count()
        _, *plain = pf.pf_lowrank_conv_bwd(x, U, V, dY, T_stash=T, need_dX=dX)
        launches = pf.pf_launch_count() - before
        assert launches == (4 if dX and R % 16 and 64 % R else 3)        # (dX reads a copy of U)
        sums = None
        for dtype in (torch.float32, torch.bfloat16):
            for accumulate in (False, True):
                for offset in (0, 1):
                    out = [torch.full((g.numel() + 1,), 0.5, dtype=dtype, device="cuda")[offset:offset + g.numel()].view(g.shape) for g in plain]
                    before = pf.pf_launch_count()
                    pf.pf_lowrank_conv_bwd(x, U, V, dY, T_stash=T, need_dX=dX, dU=out[0], dV=out[1], accumulate=accumulate, grads_f32=dtype == torch.float32)
                    if accumulate or dtype == torch.float32:
                        assert pf.pf_launch_count() - before == launches
                    torch.cuda.synchronize()
                    if sums is None:
                        sums = [o.clone() for o in out]
                        assert all(torch.equal(s.bfloat16(), g) for s, g in zip(sums, plain))
                    if dtype == torch.float32 or accumulate or offset == 0:      # (plain matrices off a 16-byte boundary take the other form)
                        assert all(torch.equal(o, ((s + 0.5) if accumulate else s).to(dtype)) for o, s in zip(out, sums)), (dX, dtype, accumulate, offset)


@pytest.mark.parametrize("N,H,W,C,R,O,without", [
    (32, 28, 28, 192, 48, 192, 2), (90, 28, 28, 192, 48, 192, 3), (28, 28, 28, 64, 24, 64, 2), (120, 28, 28, 64, 24, 64, 3), (20, 20, 20, 512, 24, 512, 2),
    (20, 28, 28, 448, 56, 448, 2), (16, 28, 28, 160, 40, 160, 2), (48, 28, 28, 160, 40, 160, 3), (130, 32, 32, 64, 32, 64, 2)])
def test_backward_without_dX_chooses_for_itself(N, H, W, C, R, O, without):
    """What dX gains does not count for a call that does not want it."""
    x, U, V, dY = (torch.zeros(*s, dtype=torch.bfloat16, device="cuda") for s in ((N, H, W, C), (3, 3, C, R), (O, R), (N, H, W, O)))
    T = torch.zeros(N, H, W, R, dtype=torch.bfloat16, device="cuda")
    before = pf.pf_launch_count()
    pf.pf_lowrank_conv_bwd(x, U, V, dY, T_stash=T, need_dX=False)
    assert pf.pf_launch_count() - before == without
    if C * R <= 160 * 48 and N < 64:
        run_conv(wl.ConvCase("no dX", N, H, W, C, R, O, wl.BF16, 93), need_dX=False)


@pytest.mark.parametrize("N,H,W,C,R,O,stride,room", [(45, 16, 16, 320, 40, 72, 1, 10154752), (140, 9, 13, 136, 24, 136, 1, 8250624),
                                                     (60, 15, 14, 40, 24, 40, 2, 6124800)])
def test_backward_in_the_least_workspace(N, H, W, C, R, O, stride, room):
    """Scratch without room for what reads less: the products that fetch pixels per tap, on rows as they lie."""
    c = wl.ConvCase("least", N, H, W, C, R, O, wl.BF16, 96, stride=stride)
    assert pf.pf_lowrank_conv_workspace(N, H, W, C, R, O, 3, 3, stride, 1, pf.PF_BF16, True) > room
    run_conv(c, bwd_room=room)
    run_conv(c, stash=False, need_dX=False, bwd_room=room)


@pytest.mark.parametrize("N,H,W,C,R,O", [(45, 16, 16, 320, 40, 72), (140, 9, 13, 136, 24, 136), (300, 7, 7, 256, 40, 64), (60, 28, 28, 128, 8, 128)])
@pytest.mark.parametrize("how", ["plain", "grads_f32", "accumulate"])
def test_flat_backward_infinities_at_the_border(N, H, W, C, R, O, how):
    """A border pixel that is no number reaches only the taps that pair it with a pixel of y: the others of its channel are what
    they are with a zero there, the other channels are untouched.  An infinity in dY likewise reaches the pixels of x that it is paired with."""
    g = torch.Generator(device="cuda").manual_seed(99)
    rand = lambda *s: torch.rand(s, generator=g, device="cuda").add_(0.25).bfloat16()       # (no zeros, no signs: infinities stay infinities)
    x, U, V, dY = rand(N, H, W, C), rand(3, 3, C, R), rand(O, R), rand(N, H, W, O)
    kw = dict(grads_f32=how == "grads_f32")

    def grads(x, dY):
        if how == "accumulate":
            kw.update(accumulate=True, dU=torch.ones_like(U), dV=torch.ones_like(V))
        return pf.pf_lowrank_conv_bwd(x, U, V, dY, **kw)[1:]

    borders = [((3, 0, 2, 1), float("inf")), ((N - 1, H - 1, 4, 7), float("inf")), ((0, 3, 0, C - 1), float("nan")), ((5, 2, W - 1, 64), float("-inf")),
               ((1, 0, 0, 2), float("inf")), ((2, H - 1, W - 1, 3), float("nan"))]
    bad, zeroed = x.clone(), x.clone()
    reached = torch.zeros(3, 3, C, dtype=torch.bool, device="cuda")
    for at, v in borders:
        bad[at], zeroed[at] = v, 0
        for ky in range(3):
            for kx in range(3):
                reached[ky, kx, at[3]] |= 0 <= at[1] - (ky - 1) < H and 0 <= at[2] - (kx - 1) < W
    (dU, dV), (dU0, dV0) = grads(bad, dY), grads(zeroed, dY)
    assert not dU[reached].isfinite().any() and torch.isinf(dU[1, 1, 1]).all()
    # fp32 sums of positive products in another order: n units in the last place of half of one each; bf16 rounds twice
    tol = N * H * W * 2.0 ** -24 + (0 if how == "grads_f32" else 2.0 ** -7)
    rest = ~reached
    assert dU[rest].isfinite().all() and ((dU[rest].double() - dU0[rest].double()).abs() <= tol * dU0[rest].double()).all()
    clean = torch.ones(C, dtype=torch.bool, device="cuda")
    clean[[at[3] for at, _ in borders]] = False
    assert torch.equal(dU[:, :, clean], dU0[:, :, clean])
    inf_dY = dY.clone()
    inf_dY[4, H - 1, 0, 5] = float("inf")
    dU, dV = grads(x, inf_dY)
    for ky in range(3):
        for kx in range(3):
            assert (dU[ky, kx].isfinite() if H - 1 + ky - 1 >= H or kx - 1 < 0 else dU[ky, kx].isinf()).all(), (ky, kx)
    assert dV[5].isinf().all() and dV[6].isfinite().all()
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("N,H,W,C,R,O,k,stride,pad,copied", [
    (60, 15, 14, 40, 24, 40, 3, 1, 1, True),        # per tap, ragged channels, a rank within one line
    (60, 14, 15, 64, 72, 72, 3, 2, 1, False),       # too few pixels once the stride is taken
    (47, 16, 16, 64, 72, 200, 3, 1, 1, True),       # just enough pixels, two rank blocks
    (46, 16, 16, 64, 72, 200, 3, 1, 1, False),
    (200, 28, 28, 72, 40, 136, 3, 1, 1, True),      # resident windows, ragged channels: one plane of U per tap
    (200, 28, 28, 128, 40, 64, 3, 1, 1, True),
    (60, 16, 16, 64, 136, 64, 1, 1, 0, True),
])
def test_forward_copies_of_the_factors(N, H, W, C, R, O, k, stride, pad, copied):
    """Rows of U and V that straddle lines are copied to a pitch of whole ones; scratch without room for that runs on the
    rows as they lie, to the same sums in the same order."""
    c = wl.ConvCase("copies", N, H, W, C, R, O, wl.BF16, 98, kh=k, kw=k, stride=stride, pad=pad)
    run_conv(c)
    d = c.generate()
    x, U, V = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V"))
    before = pf.pf_launch_count()
    y, T = pf.pf_lowrank_conv_fwd(x, U, V, stride=stride, pad=pad, want_stash=True)
    assert pf.pf_launch_count() - before == 1 + copied
    room = (T.numel() * 2 + 255) // 256 * 256
    y1, T1 = pf.pf_lowrank_conv_fwd(x, U, V, stride=stride, pad=pad, want_stash=True, workspace=torch.empty(room, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    assert torch.equal(y, y1) and torch.equal(T, T1)


@pytest.mark.parametrize("N,H,R,k,stride,forward,backward", [
    (16, 28, 40, 1, 1, 0, 0), (32, 28, 40, 1, 1, 1, 0), (32, 28, 40, 3, 2, 0, 0), (16, 28, 56, 3, 1, 0, 0), (32, 28, 56, 3, 1, 0, 0), (32, 28, 56, 5, 1, 1, 0),
    (32, 28, 72, 1, 1, 1, 0), (108, 28, 72, 3, 2, 1, 1), (16, 28, 80, 3, 1, 0, 0), (32, 28, 80, 3, 1, 1, 1), (32, 28, 80, 1, 1, 0, 0), (32, 28, 96, 3, 1, 0, 1),
    (103, 28, 24, 5, 1, 0, 0)])
def test_copies_where_they_are_worth_a_launch(N, H, R, k, stride, forward, backward):
    """One launch more where the factors, or U for dX, are copied to a pitch of whole lines, none elsewhere; the results are
    those of the rows as they lie."""
    C, O, pad = 64, 64, k // 2
    g = torch.Generator(device="cuda").manual_seed(92)
    rand = lambda *s, scale=1.0: torch.randn(s, generator=g, device="cuda").mul_(scale).bfloat16()
    x, U, V = rand(N, H, H, C), rand(k, k, C, R, scale=(k * k * C) ** -0.5), rand(O, R, scale=R ** -0.5)
    before = pf.pf_launch_count()
    y, T = pf.pf_lowrank_conv_fwd(x, U, V, stride=stride, pad=pad, want_stash=True)
    assert pf.pf_launch_count() - before == 1 + forward
    dY = rand(*y.shape)
    before = pf.pf_launch_count()
    out = pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, pad=pad, T_stash=T)
    launches = pf.pf_launch_count() - before
    before = pf.pf_launch_count()
    pf.pf_lowrank_conv_bwd(x, U, V, dY, stride=stride, pad=pad, T_stash=T, need_dX=False)
    without = pf.pf_launch_count() - before
    assert launches == 2 + backward + (1 if without == 3 or (k == 3 and stride == 1 and R < 64 and N * H * H >= 25000) else 0)
    room = (T.numel() * 2 + 255) // 256 * 256
    y1, T1 = pf.pf_lowrank_conv_fwd(x, U, V, stride=stride, pad=pad, want_stash=True, workspace=torch.empty(room, dtype=torch.uint8, device="cuda"))
    assert torch.equal(y, y1) and torch.equal(T, T1)
    d64 = lambda t: t.double().permute(0, 3, 1, 2)
    dT = (dY.double() @ V.double()).bfloat16()
    dX = torch.nn.grad.conv2d_input((N, C, H, H), U.double().permute(3, 2, 0, 1), d64(dT), stride=stride, padding=pad).permute(0, 2, 3, 1)
    assert (out[0].double() - dX).norm() <= 1e-2 * dX.norm()


@pytest.mark.parametrize("N,H,W,C,R,O,k,stride,pad", [
    (163, 16, 16, 64, 16, 64, 3, 1, 1),      # two dX tiles per block, a last block with one
    (41, 30, 30, 136, 24, 40, 3, 2, 1),      # eight per block, two column tiles (one ragged), all classes in a block
    (330, 9, 7, 72, 72, 40, 3, 2, 1),        # classes of unequal size, two rank blocks per tap
    (150, 14, 14, 64, 8, 24, 5, 3, 2),       # nine classes of one to four taps
    (310, 8, 8, 64, 136, 200, 3, 1, 1),      # dT as well: ragged k-block, two column tiles
    (300, 13, 13, 64, 16, 64, 4, 4, 0),      # stride 4: one tap per class
])
def test_several_dx_tiles_per_block(N, H, W, C, R, O, k, stride, pad):
    """Enough output tiles of dX for several in a block: accumulators and pipeline stages change hands between tiles."""
    run_conv(wl.ConvCase("dx", N, H, W, C, R, O, wl.BF16, 96, kh=k, kw=k, stride=stride, pad=pad))
