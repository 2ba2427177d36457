"""GPU parity: factorized linear forward/backward through the C ABI vs the fp64 oracle."""
import itertools

import numpy as np
import pytest
import torch

import oracle
import paper_2103_03936_b200 as pf
import pf_workloads as wl
from _gpu import ESCAPES, Guarded, assert_blocks_close, assert_close, dev, host, linear_scratch

pytestmark = pytest.mark.gpu


def run_case(case, ld_pad=0, stash=True, need_dX=True, tiny=False, blocks=False):
    d = case.generate()
    dt = case.dtype
    m, k, n, r = case.m, case.k, case.n, case.r

    def up(a, cols):
        if not ld_pad:
            return dev(a, dt)
        buf = torch.zeros((a.shape[0], cols + ld_pad), dtype=wl.to_torch(a[:1], dt).dtype, device="cuda")
        buf[:, :cols] = dev(a, dt)
        return buf[:, :cols]

    x, U, V, dY = up(d["x"], k), up(d["U"], r), up(d["V"], r), up(d["dY"], n)
    gy = Guarded((m, n), dt, ld=n + ld_pad if ld_pad else None)
    gT = Guarded((m, r), dt, ld=r + ld_pad if ld_pad else None)
    scratch = [linear_scratch(x, U, V, bwd) for bwd in (False, True)]
    out = pf.pf_lowrank_linear_fwd(x, U, V, y=gy.t, T_stash=gT.t if stash else None, workspace=scratch[0].t)
    y_ref, T_ref = oracle.linear_fwd(d["x"], d["U"], d["V"])
    dX_ref, dU_ref, dV_ref = oracle.linear_bwd(d["x"], d["U"], d["V"], d["dY"])
    gdX = Guarded((m, k), dt, ld=k + ld_pad if ld_pad else None)
    gdU = Guarded((k, r), dt, ld=r + ld_pad if ld_pad else None)
    gdV = Guarded((n, r), dt, ld=r + ld_pad if ld_pad else None)
    pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=gT.t if stash else None, need_dX=need_dX,
                             dX=gdX.t if need_dX else None, dU=gdU.t, dV=gdV.t, workspace=scratch[1].t)
    torch.cuda.synchronize()
    ab = {}
    if tiny:   # magnitude of the summands, for outputs of a handful of elements
        aw = {k_: np.abs(oracle.widen(v)) for k_, v in d.items()}
        ab["y"], ab["T"] = oracle.linear_fwd(aw["x"], aw["U"], aw["V"])
        ab["dX"], ab["dU"], ab["dV"] = oracle.linear_bwd(aw["x"], aw["U"], aw["V"], aw["dY"])
    tag = f"{case.name} {m}x{k}->{n} r{r} {dt} "
    checks = [("y", gy, y_ref)]
    if stash:
        checks.append(("T", gT, T_ref))
    if need_dX:
        checks.append(("dX", gdX, dX_ref))
    checks += [("dU", gdU, dU_ref), ("dV", gdV, dV_ref)]
    errs = {}
    for nm, g, ref in checks:
        errs[nm] = assert_close(g.t, ref, dt, tag + nm, abs_ref64=ab.get(nm))
        if blocks:   # and no 128 x 128 block of the tensor may miss the same bound
            errs[nm + " worst block"] = assert_blocks_close(g.t, ref, dt, tag + nm)
    for g in (gy, gT, gdX, gdU, gdV, *scratch):
        g.check()
    assert pf.pf_last_device_status() == 0
    return errs


GRID = [(m, k, n, r) for m, k, n, r in itertools.product((1, 7, 130), (1, 17, 100), (3, 24, 130), (1, 5, 33))]


# Outputs of the bf16 grid that may be measured against the magnitude of their summands (see
# _gpu.assert_close): single near-cancelled sums.  The count is fixed by the seeded inputs.
MAX_CANCELLED_OUTPUTS = 2


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_tiny_exhaustive_grid(dtype):
    first = len(ESCAPES)
    for idx, (m, k, n, r) in enumerate(GRID):
        run_case(wl.LinearCase(f"g{idx}", m, k, n, r, dtype, 100 + idx), tiny=True)
    took = ESCAPES[first:]
    for what, rel, ratio, err_abs in took:
        print(f"cancelled output {what}: rel {rel:.2e}, |exact|/|summands| {ratio:.2e}, err vs summands {err_abs:.2e}")
    assert len(took) <= (MAX_CANCELLED_OUTPUTS if dtype == wl.BF16 else 0), took


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
@pytest.mark.parametrize("m,k,n,r", [(257, 72, 136, 24), (300, 200, 264, 40), (129, 64, 64, 64),
                                     (1000, 328, 520, 96)])
def test_multi_tile_ragged(dtype, m, k, n, r):
    run_case(wl.LinearCase("rag", m, k, n, r, dtype, 7))


@pytest.mark.parametrize("m,k,n,r", [(2100, 200, 328, 40), (2048, 1504, 520, 376), (2500, 136, 72, 200),
                                     (4100, 72, 1000, 130), (2048, 64, 64, 256), (2304, 520, 264, 320),
                                     (2050, 100, 130, 33)])
def test_fused_chain_envelope(m, k, n, r):
    """m >= 2048 with r <= 192 takes the fused two-GEMM kernel (rank paddings 64, 128, 192; ragged
    row tile, ragged k / n tails, with and without stash and dX); the larger ranks of this list run
    as unfused products on the same batch sizes."""
    run_case(wl.LinearCase("chain", m, k, n, r, wl.BF16, 13))
    run_case(wl.LinearCase("chain", m, k, n, r, wl.BF16, 14), stash=False, need_dX=False)


@pytest.mark.parametrize("m,k,n,r", [(19500, 200, 128, 64), (40000, 136, 72, 100)])
def test_fused_chain_more_row_tiles_than_sms(m, k, n, r):
    """More 128-row tiles than SMs: the fused kernel runs as a persistent grid in which a CTA owns
    several tiles (unequal counts, a ragged last tile) and the phases of consecutive tiles overlap;
    forward (one and two output column tiles per row tile) and dX, with and without the stash."""
    run_case(wl.LinearCase("multi", m, k, n, r, wl.BF16, 19))
    run_case(wl.LinearCase("multi", m, k, n, r, wl.BF16, 20), stash=False, need_dX=False)


@pytest.mark.parametrize("m,k,n,r", [(16000, 72, 264, 520), (9000, 200, 520, 392)])
def test_wide_unfused_products_on_cta_pairs(m, k, n, r):
    """Ranks above 384 run as plain products; wide ones with many tiles use the two-CTA MMA kernel:
    a ragged last row pair, ragged column tiles and a ragged k tail, K-major and MN-major B."""
    run_case(wl.LinearCase("pairs", m, k, n, r, wl.BF16, 17))


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_leading_dimensions_and_padding_untouched(dtype):
    run_case(wl.LinearCase("ld", 200, 72, 136, 24, dtype, 8), ld_pad=8)
    run_case(wl.LinearCase("ld", 77, 33, 50, 7, dtype, 9), ld_pad=3)


@pytest.mark.parametrize("m", [20, 300, 2100, 19500])
def test_ragged_widths_at_pitches_of_whole_16_byte_pieces(m):
    """Rows that end inside a piece at pitches that TMA takes: what lies behind the last column is the caller's."""
    run_case(wl.LinearCase("ld", m, 60, 140, 28, wl.BF16, 80), ld_pad=4)
    run_case(wl.LinearCase("ld", m, 60, 144, 28, wl.BF16, 81), ld_pad=4, stash=False)


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_recompute_without_stash_and_no_dX(dtype):
    run_case(wl.LinearCase("ns", 300, 136, 72, 24, dtype, 10), stash=False)
    run_case(wl.LinearCase("nx", 300, 136, 72, 24, dtype, 11), need_dX=False)


def test_config_C1_tiny_fp32():
    run_case(wl.linear_cases()["C1"])


@pytest.mark.parametrize("name", ["C2a", "C2b", "C3i", "C3h"])
def test_configs_full_size(name):
    errs = run_case(wl.linear_cases()[name], blocks=True)
    print(name, errs)


def test_config_C3_padded_pitch():
    """LSTM shape with 16-byte-multiple row pitches (k 1500->1504, r 375->376 elements)."""
    run_case(wl.linear_cases()["C3i"], ld_pad=0)
    c = wl.linear_cases()["C3i"]
    d = c.generate()

    def padded(a, cols, ld):
        buf = torch.zeros((a.shape[0], ld), dtype=torch.bfloat16, device="cuda")
        buf[:, :cols] = dev(a, c.dtype)
        return buf[:, :cols]
    x, U, V, dY = padded(d["x"], 1500, 1504), padded(d["U"], 375, 376), padded(d["V"], 375, 376), dev(d["dY"], c.dtype)
    y, T = pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
    y_ref, _ = oracle.linear_fwd(d["x"], d["U"], d["V"])
    dX_ref, dU_ref, dV_ref = oracle.linear_bwd(d["x"], d["U"], d["V"], d["dY"])
    for got, want, nm in ((y, y_ref, "y"), (dX, dX_ref, "dX"), (dU, dU_ref, "dU"), (dV, dV_ref, "dV")):
        assert_close(got, want, c.dtype, nm)


@pytest.fixture(scope="module")
def sweep_inputs():
    c = wl.linear_cases()["C5r16"]
    x = wl.round_to(wl.normal(c.seed, 0, (c.m, c.k)), c.dtype)
    dY = wl.round_to(wl.normal(c.seed, 3, (c.m, c.n)), c.dtype)
    return x, dY, dev(x, c.dtype), dev(dY, c.dtype)


@pytest.mark.parametrize("r", [16, 128, 256, 1024])
def test_rank_sweep_full_size_sampled(sweep_inputs, r):
    """m=16384, k=n=4096: y and dX on sampled rows, dU and dV on sampled rank columns (the
    oracle computes those exactly from sliced inputs), in the configuration the bench times."""
    x_h, dY_h, x, dY = sweep_inputs
    c = wl.linear_cases()[f"C5r{r}"]
    import math
    sig = 1.0 / math.sqrt(c.k)
    U_h = wl.round_to(wl.normal(c.factor_seed, 1, (c.k, r), sig), c.dtype)
    V_h = wl.round_to(wl.normal(c.factor_seed, 2, (c.n, r), sig), c.dtype)
    U, V = dev(U_h, c.dtype), dev(V_h, c.dtype)
    y, T = pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
    torch.cuda.synchronize()
    rows = [0, 1, 127, 128, 5000, 8191, 8192, 16383]
    y_ref, T_ref = oracle.linear_fwd(x_h[rows], U_h, V_h)
    dX_ref, _, _ = oracle.linear_bwd(x_h[rows], U_h, V_h, dY_h[rows])
    for got, want, nm in ((y[rows], y_ref, "y rows"), (T[rows], T_ref, "T rows"), (dX[rows], dX_ref, "dX rows")):
        assert_close(got, want, c.dtype, nm)
        assert_blocks_close(got, want, c.dtype, nm)          # 8 sampled rows x 128 columns per block
    J = sorted({0, r // 2, r - 1})
    _, dU_ref, dV_ref = oracle.linear_bwd(x_h, U_h[:, J], V_h[:, J], dY_h)
    for got, want, nm in ((dU[:, J], dU_ref, "dU cols"), (dV[:, J], dV_ref, "dV cols")):
        assert_close(got, want, c.dtype, nm)
        assert_blocks_close(got, want, c.dtype, nm)          # 128 rows x the sampled columns per block
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_backward_is_bit_reproducible(dtype):
    c = wl.LinearCase("rep", 4096, 256, 320, 64, dtype, 12)
    d = c.generate()
    x, U, V, dY = (dev(d[k_], dtype) for k_ in ("x", "U", "V", "dY"))
    a = pf.pf_lowrank_linear_bwd(x, U, V, dY)
    b = pf.pf_lowrank_linear_bwd(x, U, V, dY)
    torch.cuda.synchronize()
    for p, q in zip(a, b):
        assert torch.equal(p, q)


def test_split_reductions_on_two_streams_do_not_interfere():
    """The slice sums of dU / dV meet at per-tile counters inside the library; launches that are in
    flight at the same time on different streams must use different counter sets."""
    cases = [wl.LinearCase("s0", 4096, 256, 320, 64, wl.BF16, 21), wl.LinearCase("s1", 3000, 384, 256, 128, wl.BF16, 22)]
    ins = []
    for c in cases:
        d = c.generate()
        ins.append(tuple(dev(d[k_], wl.BF16) for k_ in ("x", "U", "V", "dY")))
    ref = [pf.pf_lowrank_linear_bwd(*t) for t in ins]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [[], []]
    for it in range(6):
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                outs[i].append(pf.pf_lowrank_linear_bwd(*ins[i], stream=st))
    torch.cuda.synchronize()
    for i in range(2):
        for got in outs[i]:
            for p, q in zip(got, ref[i]):
                assert torch.equal(p, q)
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
def test_empty_batch(dtype):
    tdt = torch.float32 if dtype == wl.F32 else torch.bfloat16
    x = torch.empty((0, 16), dtype=tdt, device="cuda")
    U = torch.ones((16, 4), dtype=tdt, device="cuda")
    V = torch.ones((8, 4), dtype=tdt, device="cuda")
    y = pf.pf_lowrank_linear_fwd(x, U, V)
    assert y.shape == (0, 8)
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, torch.empty((0, 8), dtype=tdt, device="cuda"),
                                          dU=torch.full((16, 4), 3.0, dtype=tdt, device="cuda"),
                                          dV=torch.full((8, 4), 3.0, dtype=tdt, device="cuda"))
    torch.cuda.synchronize()
    assert torch.all(dU == 0) and torch.all(dV == 0)


def test_invalid_arguments_raise_not_launch():
    x = torch.zeros((4, 8), dtype=torch.bfloat16, device="cuda")
    U = torch.zeros((8, 2), dtype=torch.bfloat16, device="cuda")
    V = torch.zeros((6, 2), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(pf.PfError) as e:
        pf.pf_lowrank_linear_fwd(x, U, V, workspace=torch.empty(8, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 3


@pytest.mark.parametrize("m,k,n,r", [(128, 32, 64, 64), (129, 36, 132, 68), (1, 4, 4, 4), (257, 100, 260, 33), (64, 1000, 72, 129),
                                     (2500, 64, 200, 24), (300, 2052, 1028, 260)])
def test_fp32_products_on_tensor_cores(m, k, n, r):
    """fp32 storage through the split-operand kernel: edges of the 128-row, 64- and 128-column tiles and of the
    32-element k-blocks, whole and sliced contractions, ragged pitches; held to fp32 accuracy, ten times
    tighter than the fp32 tolerance asks."""
    c = wl.LinearCase("f32tc", m, k, n, r, wl.F32, 23)
    errs = run_case(c)
    assert max(errs.values()) <= 1e-5, errs
    run_case(wl.LinearCase("f32tc", m, k, n, r, wl.F32, 24), stash=False, need_dX=False)


@pytest.mark.parametrize("m,k,n,r", [(1, 1, 1, 1), (1, 17, 33, 15), (8, 256, 64, 16), (9, 300, 100, 17), (16, 1000, 31, 40), (20, 1500, 600, 375),
                                     (25, 2049, 65, 33), (32, 513, 257, 129), (32, 64, 96, 1000)])
def test_few_rows_forward(m, k, n, r):
    """Up to 32 rows: the kernels without re-pitch copies; edges of the 8-row, 16-column and 32-row blocks, contractions
    shared by clusters, odd pitches, bias and activation."""
    c = wl.LinearCase("few", m, k, n, r, wl.BF16, 27)
    for pad in (0, 3):
        d = c.generate()
        def up(a, cols):
            buf = torch.zeros((a.shape[0], cols + pad), dtype=torch.bfloat16, device="cuda")
            buf[:, :cols] = dev(a, c.dtype)
            return buf[:, :cols]
        gy, gT = Guarded((m, n), c.dtype, ld=n + pad), Guarded((m, r), c.dtype, ld=r + pad)
        b = wl.round_to(wl.normal(28, 7, (n,), 0.5), c.dtype)
        pf.pf_lowrank_linear_fwd_act(up(d["x"], k), up(d["U"], r), up(d["V"], r), bias=dev(b, c.dtype), act=pf.PF_ACT_RELU, y=gy.t, T_stash=gT.t)
        torch.cuda.synchronize()
        y_ref, T_ref = oracle.linear_fwd_act(d["x"], d["U"], d["V"], b, relu=True)
        assert_close(gT.t, T_ref, c.dtype, "few rows T")
        if np.linalg.norm(y_ref) > 0:
            assert_close(gy.t, y_ref, c.dtype, "few rows y")
        gy.check()
        gT.check()
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("m,k,n,r", [(14001, 72, 136, 136), (2331, 128, 64, 72), (9600, 64, 64, 16)])
def test_row_tiles_of_96(m, k, n, r):
    """Batches whose 128-row tiles would leave SMs idle run the fused kernel on 96-row tiles: guard bands, ragged last
    tiles, both directions, padded pitches."""
    run_case(wl.LinearCase("rows", m, k, n, r, wl.BF16, 29))
    run_case(wl.LinearCase("rows", m, k, n, r, wl.BF16, 30), ld_pad=8)


def test_re_pitch_copies_beyond_two_to_the_31_pieces():
    """Ragged operands of more than 2^31 pieces of 16 bytes are copied in several launches: 34 GB of zeros with a few small
    integers around the seams, so that every result is exact."""
    m, k, n = 4100, 4194297, 8
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    x = torch.zeros((m, k), dtype=torch.bfloat16, device="cuda")
    U = torch.randint(-3, 4, (k, n), device="cuda").to(torch.bfloat16)
    V = torch.eye(n, dtype=torch.bfloat16, device="cuda")
    want = torch.zeros((m, n), dtype=torch.bfloat16, device="cuda")
    cols = torch.tensor([0, 1, 7, 8, 63, 64, k // 2, k - 9, k - 2, k - 1], device="cuda")
    for row in (0, 1, 2047, 2048, 4094, 4095, 4096, 4099):
        x[row, cols] = torch.randint(-3, 4, (len(cols),), device="cuda").to(torch.bfloat16)
        want[row] = (x[row, cols].float() @ U[cols].float()).to(torch.bfloat16)
    launches = pf.pf_launch_count()
    y = pf.pf_lowrank_linear_fwd(x, U, V)
    assert pf.pf_launch_count() - launches == 3
    assert torch.equal(y, want)
    assert pf.pf_last_device_status() == 0
    del x, y
    torch.cuda.empty_cache()


@pytest.mark.parametrize("m,k,n,r", [(130, 64, 1, 16), (300, 64, 63, 16), (300, 72, 129, 40), (160, 64, 200, 392), (4200, 64, 2561, 256)])
@pytest.mark.parametrize("base,pad", [(0, 1), (1, 0), (3, 5), (4, 4), (7, 2)])
def test_output_rows_of_any_alignment(m, k, n, r, base, pad):
    """Output rows that start anywhere and whose pitch is anything hold, bit for bit, what rows on 16-byte boundaries
    hold, and nothing around them is touched (single tiles, CTA pairs, y and the stash)."""
    d = wl.LinearCase("rows", m, k, n, r, wl.BF16, 71).generate()
    x, U, V = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V"))

    def rows(cols, start, ld):
        buf = torch.full((start + m * ld + 64,), -7.0, dtype=torch.bfloat16, device="cuda")
        return buf, buf[start:start + m * ld].view(m, ld)[:, :cols]

    _, y0 = rows(n, 64, (n + 7) // 8 * 8)
    _, T0 = rows(r, 64, (r + 7) // 8 * 8)
    pf.pf_lowrank_linear_fwd(x, U, V, y=y0, T_stash=T0)
    by, y1 = rows(n, 64 + base, n + pad)
    bT, T1 = rows(r, 64 + base, r + pad + (r + pad + 1) % 2)        # an odd pitch: the second copy
    pf.pf_lowrank_linear_fwd(x, U, V, y=y1, T_stash=T1)
    torch.cuda.synchronize()
    assert_close(y0, oracle.linear_fwd(d["x"], d["U"], d["V"])[0], wl.BF16, f"{m}x{k}->{n} r{r} y")
    for want, got, buf in ((y0, y1, by), (T0, T1, bT)):
        assert torch.equal(want, got)
        got.fill_(-7.0)
        assert bool((buf == -7.0).all()), "written outside the rows"
    assert pf.pf_last_device_status() == 0


@pytest.mark.parametrize("m,k,n,r", [(1100, 256, 264, 40), (1216, 264, 256, 40), (4096, 256, 256, 256), (2050, 520, 520, 200), (700, 2056, 1032, 264),
                                     (2500, 1032, 4104, 520)])
def test_whole_and_split_contractions_and_pairs(m, k, n, r):
    """Either side of the lengths from which contractions are split, and of the sizes from which products run on CTA
    pairs; dU and dV split by themselves beside a product that is whole."""
    run_case(wl.LinearCase("forms", m, k, n, r, wl.BF16, 72), blocks=True)


@pytest.mark.parametrize("m,k,n,r", [(300, 136, 264, 40), (1100, 72, 1032, 200), (1000, 520, 520, 72), (1300, 104, 136, 24), (2320, 984, 2872, 440)])
def test_orders_of_the_unfused_backward(m, k, n, r):
    """Two launches (dV beside G, dU beside dX), three (dU, dV and dX behind G, whole and split) and G and dX on CTA pairs; with and
    without dX and the stash."""
    run_case(wl.LinearCase("order", m, k, n, r, wl.BF16, 82), blocks=m > 128)
    run_case(wl.LinearCase("order", m, k, n, r, wl.BF16, 83), stash=False, need_dX=False)


@pytest.mark.parametrize("m,k,n,r", [(2048, 516, 2052, 1028), (2048, 2052, 516, 1028), (2100, 520, 3080, 520)])
def test_reductions_that_do_not_fit_the_machine_together(m, k, n, r):
    """The tiles of dU and dV are more than the SMs; each is split by itself, within the workspace that is asked for."""
    run_case(wl.LinearCase("wide", m, k, n, r, wl.BF16, 78), blocks=True)
    run_case(wl.LinearCase("wide", m, k, n, r, wl.BF16, 79), stash=False, need_dX=False)


@pytest.mark.parametrize("m,k,n,r", [(1, 8, 8, 8), (5, 512, 136, 24), (32, 512, 1032, 192), (33, 1536, 264, 64), (129, 72, 4104, 136), (2047, 1536, 128, 16)])
def test_fused_forward_of_smaller_batches(m, k, n, r):
    """Forward with k <= 1536 (512 up to 32 rows) and r <= 192: one launch; one column more, a rank more or a stash that TMA
    cannot write take the unfused kernels."""
    case = wl.LinearCase("fused small", m, k, n, r, wl.BF16, 73)
    run_case(case, blocks=m > 100)
    d = case.generate()
    x, U, V = (dev(d[k_], wl.BF16) for k_ in ("x", "U", "V"))
    before = pf.pf_launch_count()
    pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
    assert pf.pf_launch_count() - before == 1
    before = pf.pf_launch_count()
    pf.pf_lowrank_linear_fwd(x, U, V, T_stash=Guarded((m, r), wl.BF16, ld=r + 4).t)
    assert pf.pf_launch_count() - before == 2


@pytest.mark.parametrize("m,k,n,r", [(32, 520, 136, 24), (40, 1544, 136, 24), (300, 512, 136, 200)])
def test_forward_beyond_the_fused_sizes(m, k, n, r):
    case = wl.LinearCase("unfused small", m, k, n, r, wl.BF16, 74)
    run_case(case)
    d = case.generate()
    before = pf.pf_launch_count()
    pf.pf_lowrank_linear_fwd(*(dev(d[k_], wl.BF16) for k_ in ("x", "U", "V")))
    assert pf.pf_launch_count() - before == 2


@pytest.mark.parametrize("m,k,n,r", [(1030, 260, 260, 68), (516, 1540, 1030, 128), (2048, 128, 516, 132)])
def test_fp32_wide_tiles_in_more_slices(m, k, n, r):
    """fp32 reductions that take 128-column tiles in more slices instead of 64-column ones: ragged tiles, same accuracy."""
    errs = run_case(wl.LinearCase("f32wide", m, k, n, r, wl.F32, 75))
    assert max(errs.values()) <= 1e-5, errs


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
@pytest.mark.parametrize("m,k,n,r", [(1, 1, 1, 1), (16, 32, 16, 32), (17, 33, 17, 31), (64, 256, 256, 32), (128, 128, 128, 32), (113, 100, 7, 31), (128, 5, 128, 2), (40, 24, 16, 8)])
def test_smallest_layers_in_one_launch_each_way(dtype, m, k, n, r):
    """Up to 128 rows, k and n up to 256 (bf16: 128), r up to 32: edges of the 16- and 32-wide tiles and of the cluster, any
    pitch; the backward is one launch, and so is the fp32 forward."""
    if dtype == wl.BF16:
        k, n = min(k, 128), min(n, 128)
    case = wl.LinearCase("tiny", m, k, n, r, dtype, 76)
    run_case(case, ld_pad=0, tiny=True)
    run_case(case, ld_pad=3, tiny=True, need_dX=False)
    d = case.generate()
    x, U, V, dY = (dev(d[k_], dtype) for k_ in ("x", "U", "V", "dY"))
    before = pf.pf_launch_count()
    _, T = pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
    assert dtype == wl.BF16 or pf.pf_launch_count() - before == 1
    before = pf.pf_launch_count()
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
    assert pf.pf_launch_count() - before == 1
    # fp32 gradients are the same sums, unrounded; accumulating adds to them once
    gU, gV = torch.ones_like(dU, dtype=torch.float32), torch.ones_like(dV, dtype=torch.float32)
    pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T, dU=gU, dV=gV, grads_f32=True)
    assert torch.equal(gU.to(dU.dtype), dU) and torch.equal(gV.to(dV.dtype), dV)
    aU, aV = torch.ones_like(gU), torch.ones_like(gV)
    pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T, dU=aU, dV=aV, grads_f32=True, accumulate=True)
    assert torch.equal(aU, gU + 1) and torch.equal(aV, gV + 1)
    bU, bV = torch.ones_like(dU), torch.ones_like(dV)
    pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T, dU=bU, dV=bV, accumulate=True)
    assert torch.equal(bU, (gU + 1).to(dU.dtype)) and torch.equal(bV, (gV + 1).to(dV.dtype))


def test_smallest_layers_with_infinities_and_nan():
    """What is not finite reaches the outputs it belongs to and no others."""
    m, k, n, r = 40, 64, 48, 16
    for dtype in (torch.float32, torch.bfloat16):
        x, U = torch.ones(m, k, device="cuda", dtype=dtype), torch.ones(k, r, device="cuda", dtype=dtype)
        V, dY, T = torch.ones(n, r, device="cuda", dtype=dtype), torch.ones(m, n, device="cuda", dtype=dtype), torch.ones(m, r, device="cuda", dtype=dtype)
        dY[3, 5], T[7, 2], x[9, 11] = float("inf"), float("nan"), float("-inf")
        dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
        assert torch.isinf(dX[3]).all() and torch.isfinite(dX[torch.arange(m, device="cuda") != 3]).all()
        assert torch.isnan(dV[:, 2]).all() and torch.isinf(dV[5, 0]) and torch.isfinite(dV[6, 0])
        assert (dU[11].isinf() | dU[11].isnan()).all() and torch.isinf(dU[0]).all()


def test_smallest_layers_infinite_factor_and_a_ragged_batch():
    """An infinity in V makes its column of dY V and of dU infinite; the rows that pad the batch to whole tiles add nothing."""
    m, k, n, r = 41, 64, 48, 16
    for dtype in (torch.float32, torch.bfloat16):
        x, U, V, dY, T = (torch.ones(s, device="cuda", dtype=dtype) for s in ((m, k), (k, r), (n, r), (m, n), (m, r)))
        V[5, 3] = float("inf")
        dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, dY, T_stash=T)
        assert torch.isposinf(dX).all() and torch.isposinf(dU[:, 3]).all()
        assert (dU[:, 4] == m * n).all() and (dV == m).all()


@pytest.mark.parametrize("m,k,r", [(300, 512, 24), (300, 512, 33), (20, 512, 64), (2047, 136, 40), (2048, 136, 40), (5000, 136, 129),
                                   (19500, 72, 33), (18000, 3600, 72)])
def test_fused_forward_infinite_input_and_a_ragged_rank(m, k, r):
    """An infinity in x makes its row of x U and of y infinite, whatever the rank is padded to and however many rows there are:
    the single-tile, the persistent and the pipelined form of the fused kernel, with and without a bias, and beyond L2."""
    n = 136
    x, U, V = (torch.ones(s, device="cuda", dtype=torch.bfloat16) for s in ((m, k), (k, r), (n, r)))
    x[7, 11] = float("inf")
    rest = torch.arange(m, device="cuda") != 7
    for y in (pf.pf_lowrank_linear_fwd(x, U, V), pf.pf_lowrank_linear_fwd_act(x, U, V, bias=torch.zeros(n, device="cuda", dtype=torch.bfloat16))):
        assert torch.isposinf(y[7]).all() and (y[rest] == float((torch.tensor(float(k)).bfloat16().float() * r).bfloat16())).all()


def test_fused_backward_infinite_gradient_and_a_ragged_rank():
    """The same for an infinity in dY: its row of dX is infinite, the other rows are what they are without it."""
    m, k, n, r = 2100, 1032, 264, 40
    x, U, V, dY = (torch.ones(s, device="cuda", dtype=torch.bfloat16) for s in ((m, k), (k, r), (n, r), (m, n)))
    dY[7, 11] = float("inf")
    dX, _, _ = pf.pf_lowrank_linear_bwd(x, U, V, dY)
    rest = torch.arange(m, device="cuda") != 7
    assert torch.isposinf(dX[7]).all() and (dX[rest] == float((torch.tensor(float(n)).bfloat16().float() * r).bfloat16())).all()


@pytest.mark.parametrize("m,k,n,r", [(2049, 136, 1032, 64), (3499, 136, 1032, 72), (3500, 136, 1032, 72), (2100, 1032, 1024, 40), (16300, 72, 264, 16), (12000, 72, 1032, 16)])
def test_backward_schedules(m, k, n, r):
    """Either side of the sizes from which the backward's fused kernel is used, and from which dV runs beside it."""
    run_case(wl.LinearCase("schedule", m, k, n, r, wl.BF16, 77), blocks=True)


@pytest.mark.parametrize("m", [2417, 2419, 3224, 3225])
def test_copies_of_x_around_the_lines_of_their_two_forms(m):
    """188 pieces of 16 bytes a row: 454 396 and 454 772 pieces, 606 112 and 606 300, either side of 12 and 16 blocks for each of
    148 SMs.  Every row arrives whole: rows that are one power of two each make x U exact."""
    k, r, n = 1500, 64, 64
    g = torch.Generator(device="cuda").manual_seed(m)
    scale = torch.randint(-3, 4, (m, 1), generator=g, device="cuda").float().exp2()
    x = (scale * torch.ones(m, k, device="cuda")).bfloat16()
    x[:, ::3] *= -1
    U = torch.zeros(k, r, device="cuda")
    U[torch.arange(k, device="cuda"), torch.arange(k, device="cuda") % r] = 1.0
    V = torch.eye(n, r, device="cuda").bfloat16()
    y, T = pf.pf_lowrank_linear_fwd(x, U.bfloat16(), V, want_stash=True)
    want = x.double() @ U.double()          # at most 24 summands of one magnitude: exact in fp32 and in bf16
    assert torch.equal(T.double(), want) and torch.equal(y.double(), want)
