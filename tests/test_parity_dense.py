"""GPU parity of the densified tensor-core SpMM (128 x 64 tiles of A expanded in shared memory).

Taken by a default plan of a BF16 matrix with at least 2,048 rows and columns and enough entries.
Integer inputs (exact in BF16, partial sums below 2^24) match the oracle bit for bit; random
ones are held to the FP32 tolerance against the oracle on the BF16-rounded operands.
"""
import numpy as np
import pytest

import gen
import oracle
from _util import assert_within, dev

pytestmark = pytest.mark.gpu
TOL32 = 1e-5


@pytest.fixture(scope="module")
def gb():
    import paper_2604_27985_gb300 as g

    return g


def bf16(x):
    import torch

    return dev(oracle.bf16_round(x).view(np.int16)).view(torch.bfloat16)


def matrix(M, K, seed, lo=0.8, hi=1.0):
    """Rows of lo * K to hi * K entries, some empty, one full."""
    lengths = np.random.default_rng(seed).integers(int(lo * K), int(hi * K) + 1, M)
    lengths[::97] = 0
    lengths[5] = K
    return gen.csr_from_lengths(lengths, K, seed=seed)


# Nearly full rows, so that small matrices take the path (and tiles overflow their entry slots).
# Tile edges: M around a multiple of 128, K around one of 64 and of 256 (an accumulator), every
# feature tile (64, 128, 256, two of 256) full and cut
SHAPES = [(2048, 2048, 64), (2049, 2111, 72), (2175, 2049, 128), (2176, 2304, 136), (2500, 2305, 256),
          (3001, 2624, 264), (2100, 4099, 512)]


@pytest.mark.parametrize("M,K,N", SHAPES)
def test_dense_integers_bit_exact(gb, M, K, N):
    A = matrix(M, K, 700 + N)
    vals, B = gen.vals_int(A.nnz, 701), gen.dense_int(K, N, 702)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(vals), K)
    before = gb.launch_count()
    C = plan.execute(bf16(B))
    assert gb.launch_count() - before == 2  # the tile kernel and the marked rows
    plan.check()
    want, _ = oracle.spmm(A.rowptr, A.colidx, vals, B)
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)


def test_dense_sparse_tiles(gb):
    """12% of entries, all in the even 64-column tiles of the first 4,096 columns and in a few
    others: tiles below a slot's size, tiles with no entry, rows with none."""
    rng = np.random.default_rng(705)
    M, K = 6000, 6000
    cand = np.concatenate([np.arange(t, t + 64) for t in range(0, 4096, 128)] + [np.arange(5900, 6000)])
    rows, cols = [], []
    for r in range(M):
        c = cand[rng.random(cand.size) < 0.34] if r % 50 else cand[:0]
        rows.append(np.full(c.size, r))
        cols.append(c)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    vals, B = gen.vals_int(rows.size, 706), gen.dense_int(K, 256, 707)
    A = gen.csr_from_triplets(M, K, rows, cols, vals)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(vals), K)
    before = gb.launch_count()
    C = plan.execute(bf16(B))
    assert gb.launch_count() - before == 2
    plan.check()
    want, _ = oracle.spmm(A.rowptr, A.colidx, vals, B)
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)


def test_dense_random_padded_and_unaligned(gb):
    import torch

    A = matrix(2200, 2500, 710, 0.4, 0.8)
    B = gen.dense_normal(2500, 200, 711)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(A.vals), 2500)
    ref, sc = oracle.spmm(A.rowptr, A.colidx, oracle.bf16_decode(oracle.bf16_round(A.vals)),
                          oracle.bf16_decode(oracle.bf16_round(B)))
    wide = torch.zeros((2500, 232), dtype=torch.bfloat16, device="cuda")
    wide[:, :200] = bf16(B)
    for ld in (200, 204, 207):  # 32-byte, 16-byte and 4-byte aligned rows of C
        full = torch.full((2200, ld), 7.0, device="cuda")
        C = plan.execute(wide[:, :200], out=full[:, :200])
        assert_within(C.cpu().numpy(), ref, sc, TOL32, f"ld {ld}")
        assert bool((full[:, 200:] == 7.0).all())
    plan.check()


def test_dense_infinities_and_nan_stay_in_their_rows(gb):
    """An infinity or NaN in a B row reaches only the rows of C that store an entry there."""
    A = matrix(2304, 2112, 720)
    vals, B = gen.vals_int(A.nnz, 721), gen.dense_int(2112, 64, 722)
    B[100, 3], B[2000, 60] = np.inf, np.nan
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(vals), 2112)
    C = plan.execute(bf16(B)).cpu().numpy()
    plan.check()
    Z = B.copy()
    Z[100, 3] = Z[2000, 60] = 0
    want, _ = oracle.spmm(A.rowptr, A.colidx, vals, Z)
    rows = np.repeat(np.arange(A.M), np.diff(A.rowptr))
    hit_inf, hit_nan = np.zeros(A.M, bool), np.zeros(A.M, bool)
    hit_inf[rows[A.colidx == 100]] = True
    hit_nan[rows[A.colidx == 2000]] = True
    assert hit_inf.any() and hit_nan.any() and not hit_inf.all()
    assert np.array_equal(~np.isfinite(C[:, 3]), hit_inf) and np.array_equal(np.isnan(C[:, 60]), hit_nan)
    C[hit_inf, 3], C[hit_nan, 60] = want[hit_inf, 3], want[hit_nan, 60]
    assert np.array_equal(C.astype(np.float64), want)


def test_dense_plan_under_capture(gb):
    """A plan's executions replay from a CUDA graph (their scratch is the graph's)."""
    import torch

    A = matrix(2048, 2048, 725)
    vals = gen.vals_int(A.nnz, 726)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(vals), 2048)
    b, out = torch.zeros((2048, 128), dtype=torch.bfloat16, device="cuda"), torch.empty((2048, 128), device="cuda")
    plan.execute(b, out=out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _, n = launches(gb, lambda: plan.execute(b, out=out))
    assert n == 2
    for seed in (727, 728):
        B = gen.dense_int(2048, 128, seed)
        b.copy_(bf16(B))
        graph.replay()
        want, _ = oracle.spmm(A.rowptr, A.colidx, vals, B)
        assert np.array_equal(out.cpu().numpy().astype(np.float64), want)
    plan.check()


def test_dense_bounded_wait_reports_timeout(gb):
    """A tile whose B rows never arrive: the waits give up, the plan reports the timeout, and
    the block's rows are computed again on the CUDA cores."""
    A = matrix(2048, 2048, 730)
    vals, B = gen.vals_int(A.nnz, 731), gen.dense_int(2048, 64, 732)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(vals), 2048)
    want, _ = oracle.spmm(A.rowptr, A.colidx, vals, B)
    plan.test_withhold(5)
    C = plan.execute(bf16(B))
    with pytest.raises(gb.GbspError, match="TIMEOUT"):
        plan.check()
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)
    plan.test_withhold(-1)
    C = plan.execute(bf16(B))
    plan.check()
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("N,ld,off", [(264, 264, 0), (260, 260, 0), (260, 264, 0), (264, 272, 4), (264, 268, 0)])
def test_dense_plan_without_dense_windows_takes_any_operand(gb, N, ld, off):
    """Columns congruent to the row modulo 11: 9% of entries and no 16 x 8 block of 14.  Such a plan
    takes any width, leading dimension and alignment of B; whole tiles only those of 16 bytes."""
    import torch

    M, K = 9000, 3400
    rows = [np.arange(r % 11, K, 11, dtype=np.int32) for r in range(11)]
    rowptr = np.concatenate([[0], np.cumsum([rows[r % 11].size for r in range(M)])]).astype(np.int32)
    colidx = np.concatenate([rows[r % 11] for r in range(M)])
    vals, B = gen.vals_int(colidx.size, 734), gen.dense_int(K, N, 735)
    plan = gb.TcPlan(dev(rowptr), dev(colidx), bf16(vals), K)
    assert plan.info()["dense_windows"] == 0
    flat = torch.zeros(off + K * ld, dtype=torch.bfloat16, device="cuda")
    b = flat[off:].view(K, ld)[:, :N]
    b.copy_(bf16(B))
    full = torch.full((M + 1, N + 4), 7.0, device="cuda")
    C, n = launches(gb, lambda: plan.execute(b, out=full[:M, :N]))
    plan.check()
    want, _ = oracle.spmm(rowptr, colidx, vals, B)
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)
    assert bool((full[:, N:] == 7.0).all()) and bool((full[M] == 7.0).all())
    assert (n == 2) == (ld == N == 264)  # the tile kernel and the marked rows


def test_dense_plan_refuses_null_operands(gb):
    """Null B or C data is an argument error that launches nothing, as on the CSR kernels."""
    import ctypes

    from paper_2604_27985_gb300 import ops

    A = matrix(2048, 2048, 736)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(gen.vals_int(A.nnz, 737)), 2048)
    b = bf16(gen.dense_int(2048, 64, 738))
    for null in (0, 1):
        d = [ops._dense(b), ops._dense(b.float())]
        d[null].data = None
        st, n = launches(gb, lambda: ops.lib.gbsp_plan_execute(plan._h, *(ctypes.byref(x) for x in d), None))
        assert st == -1 and n == 0


def launches(gb, f):
    before = gb.launch_count()
    out = f()
    return out, gb.launch_count() - before


@pytest.mark.parametrize("M,K,N", [(12001, 2049, 128), (12100, 2111, 136), (12032, 2304, 264)])
def test_dense_without_a_plan(gb, M, K, N):
    """AUTO on a BF16 matrix regroups per call: the row statistics, one launch for that, and
    the two of a plan."""
    A = matrix(M, K, 740 + N, 0.25, 0.4)
    vals, B = gen.vals_int(A.nnz, 741), gen.dense_int(K, N, 742)
    rp, ci, v, b = dev(A.rowptr), dev(A.colidx), bf16(vals), bf16(B)
    C, n = launches(gb, lambda: gb.spmm(rp, ci, v, b))
    assert n == 4
    want, _ = oracle.spmm(A.rowptr, A.colidx, vals, B)
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want)


def test_dense_without_a_plan_any_column_order(gb):
    """Rows with repeated or unordered columns (sums of repeats, any order) go to the CUDA cores
    with their block of 128 rows; under capture, and with a chosen variant, nothing is regrouped."""
    import torch

    A = matrix(12032, 2304, 750, 0.25, 0.4)
    ci = A.colidx.copy()
    for r in (1, 700, 701):  # blocks 0 and 5
        ci[A.rowptr[r]:A.rowptr[r + 1]] = ci[A.rowptr[r]:A.rowptr[r + 1]][::-1]
    ci[A.rowptr[12031]] = ci[A.rowptr[12031] + 1]  # a repeat, in the last block
    vals, B = gen.vals_int(A.nnz, 751), gen.dense_int(2304, 128, 752)
    want, _ = oracle.spmm(A.rowptr, ci, vals, B)
    rp, c, v, b = dev(A.rowptr), dev(ci), bf16(vals), bf16(B)
    C, n = launches(gb, lambda: gb.spmm(rp, c, v, b))
    assert n == 4 and np.array_equal(C.cpu().numpy().astype(np.float64), want)
    C, n = launches(gb, lambda: gb.spmm(rp, c, v, b, variant="rowsplit"))
    assert n == 1 and np.array_equal(C.cpu().numpy().astype(np.float64), want)
    out = torch.zeros((12032, 128), device="cuda")
    graph = torch.cuda.CUDAGraph()
    gb.auto_forget()  # (a pattern unknown under capture takes the row split)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        _, n = launches(gb, lambda: gb.spmm(rp, c, v, b, out=out))
    assert n == 1
    graph.replay()
    assert np.array_equal(out.cpu().numpy().astype(np.float64), want)


def test_entries_near_2_to_the_31_stay_on_the_csr_kernels(gb):
    """Whole tiles count entries in 32 bits and look past the last one: 1,000 entries short of 2^31 - 1
    AUTO takes the row split (the statistics and one launch).  Full rows of ones: column sums."""
    import torch

    n = 46341
    nnz = 2**31 - 1 - 1000
    last = nnz - (n - 1) * n
    rowptr = torch.arange(n + 1, device="cuda", dtype=torch.int64) * n
    rowptr[n] = nnz
    colidx = torch.arange(n, device="cuda", dtype=torch.int32).repeat(n)[:nnz]
    vals = torch.ones(nnz, device="cuda", dtype=torch.bfloat16)
    B = gen.dense_int(n, 128, 756)
    C, k = launches(gb, lambda: gb.spmm(rowptr.int(), colidx, vals, bf16(B)))
    C = C.cpu().numpy().astype(np.float64)
    assert np.array_equal(C[:-1], np.broadcast_to(B.sum(0, dtype=np.float64), (n - 1, 128)))
    assert np.array_equal(C[-1], B[:last].sum(0, dtype=np.float64))
    assert k == 2


@pytest.mark.parametrize("one_sign", [False, True])
@pytest.mark.parametrize("M,K,N,density,whole", [(19000, 5000, 128, 0.10, False), (19000, 5000, 128, 0.20, True),
                                                 (12000, 3000, 256, 0.11, False), (12000, 6400, 256, 0.08, True),
                                                 (19456, 3000, 256, 0.30, True), (9728, 8192, 320, 0.05, True)])
def test_dense_without_a_plan_is_as_exact_as_the_row_split(gb, M, K, N, density, whole, one_sign):
    """Whole tiles are taken without a plan only where their error against 64 bits is the row split's or less
    (the rule's model of both errors holds within 4%).  With values and B of one sign the accumulators' losses
    add up: at N = 128, where the row split is at its best, that may cost up to 1.3 of its error."""
    import torch

    g = torch.Generator("cuda").manual_seed(744)
    n = round(density * K)
    at = torch.rand(M, K, device="cuda", generator=g).topk(n, 1).indices.sort(1).values
    rp, ci = torch.arange(M + 1, dtype=torch.int32, device="cuda") * n, at.int().reshape(-1).contiguous()
    v = (torch.rand(M * n, device="cuda", generator=g) * 2 - 1).bfloat16()
    b = torch.randn(K, N, device="cuda", generator=g).bfloat16()
    if one_sign:
        v, b = v.abs(), b.abs()
    C, k = launches(gb, lambda: gb.spmm(rp, ci, v, b))
    want = torch.sparse_csr_tensor(rp, ci, v.double(), size=(M, K)) @ b.double()
    error = lambda x: float((x.double() - want).norm() / want.norm())
    assert (k == 4) == whole
    assert error(C) <= (1.3 if one_sign and N == 128 else 1.04) * error(gb.spmm(rp, ci, v, b, variant="rowsplit"))


@pytest.mark.parametrize("M,K,N,density,whole", [(12000, 3072, 64, 0.08, False), (12000, 6144, 128, 0.08, False),
                                                 (12000, 3072, 64, 0.12, True), (9000, 3072, 264, 0.08, True)])
def test_dense_plan_is_as_exact_as_its_blocks(gb, M, K, N, density, whole):
    """A plan takes whole tiles only where their error against 64 bits is that of its blocks and CSR residual
    (here a fifth of the entries in blocks at 8%, three quarters at 12%) or less."""
    import torch

    g = torch.Generator("cuda").manual_seed(745)
    n = round(density * K)
    at = torch.rand(M, K, device="cuda", generator=g).topk(n, 1).indices.sort(1).values
    rp, ci = torch.arange(M + 1, dtype=torch.int32, device="cuda") * n, at.int().reshape(-1).contiguous()
    v = (torch.rand(M * n, device="cuda", generator=g) * 2 - 1).bfloat16()
    b = torch.randn(K, N, device="cuda", generator=g).bfloat16()
    plan, blocks = gb.TcPlan(rp, ci, v, K), gb.TcPlan(rp, ci, v, K, threshold=14)
    C, other = plan.execute(b), blocks.execute(b)
    plan.check()
    blocks.check()
    want = torch.sparse_csr_tensor(rp, ci, v.double(), size=(M, K)) @ b.double()
    error = lambda x: float((x.double() - want).norm() / want.norm())
    assert torch.equal(C, other) != whole
    assert error(C) <= 1.04 * error(other)


@pytest.mark.parametrize("band", [False, True])
def test_dense_sums_of_one_sign(gb, band):
    """Values and B of one sign, where everything that an accumulator cuts off adds up: 60% of 2,304 columns, and
    rows of 600 columns in a band.  An accumulator of e entries a row is about 2.2e-9 e too small; it takes
    at most 64 here (a full tile), 1.4e-7, beside FP32 sums of up to 36 of them (below 1e-7)."""
    import torch

    if band:
        M, K = 12000, 4096
        starts = np.linspace(0, K - 600, M).astype(np.int64)
        rowptr = np.arange(M + 1, dtype=np.int32) * 600
        colidx = (starts[:, None] + np.arange(600)).astype(np.int32).ravel()
    else:
        M, K = 4000, 2304
        A = matrix(M, K, 757, 0.6, 0.6)
        rowptr, colidx = A.rowptr, A.colidx
    rng = np.random.default_rng(758)
    vals, B = rng.random(colidx.size, dtype=np.float32), np.abs(gen.dense_normal(K, 64, 759))
    plan = gb.TcPlan(dev(rowptr), dev(colidx), bf16(vals), K)
    C, n = launches(gb, lambda: plan.execute(bf16(B)))
    plan.check()
    want, _ = oracle.spmm(rowptr, colidx, oracle.bf16_decode(oracle.bf16_round(vals)),
                          oracle.bf16_decode(oracle.bf16_round(B)))
    assert n == 2
    assert np.linalg.norm(C.cpu().numpy() - want) <= 2.4e-7 * np.linalg.norm(want)


@pytest.mark.parametrize("M,K,Kd,fp8", [(2048, 2048, 64, False), (2049, 2111, 192, False), (2175, 4097, 256, False),
                                        (2100, 2304, 128, True), (2303, 2049, 256, True), (2500, 2500, 384, False)])
def test_dense_sddmm_integers_bit_exact(gb, M, K, Kd, fp8):  # (Kd = 384 in BF16: not the path)
    """One launch over whole tiles: tile edges, ranges of tiles that change their row block, 1 to 4
    accumulators, tiles past the entries loaded ahead; E4M3 with unit scales."""
    import torch

    A = matrix(M, K, 760 + Kd, 0.2, 0.45)
    svals = gen.vals_int(A.nnz, 761)
    X, Y = gen.dense_int(M, Kd, 762, -4, 4), gen.dense_int(K, Kd, 763, -4, 4)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(A.vals), K)
    want, _ = oracle.sddmm(A.rowptr, A.colidx, svals, X, Y)
    if fp8:
        one = lambda n: torch.ones(n, device="cuda")
        f = lambda: plan.sddmm(dev(svals), dev(oracle.e4m3_round(X)), dev(oracle.e4m3_round(Y)), x_scale=one(M), y_scale=one(K))
    else:
        f = lambda: plan.sddmm(dev(svals), bf16(X), bf16(Y))
    out, n = launches(gb, f)
    plan.check()
    assert (n == 1) == (Kd != 384)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("fp8,M,K,n,stride,step", [(True, 19456, 16384, 514, 31, 7), (False, 9728, 8192, 287, 28, 5)])
def test_plan_keeps_no_tiles_that_it_would_not_take(gb, fp8, M, K, n, stride, step):
    """Where only a BF16 SpMM would take whole tiles (3.1% of entries), an E4M3 plan holds its copies of the pattern,
    the positions and the values, 13 bytes per entry, and not the tiles' 8 beside them; a BF16 plan 14, and
    not the tiles' 10, where they would pay at 512 features and not at 256 (3.5%)."""
    import torch

    ci = (torch.arange(n, device="cuda") * stride + torch.arange(M, device="cuda")[:, None] * step % stride).int().reshape(-1)
    rp = torch.arange(M + 1, dtype=torch.int32, device="cuda") * n
    v = torch.ones(M * n, device="cuda")
    v = v.to(torch.float8_e4m3fn).view(torch.uint8) if fp8 else v.bfloat16()
    s = torch.ones(M, device="cuda") if fp8 else None
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = gb.TcPlan(rp, ci, v, K, row_scale=s)
    used = before - torch.cuda.mem_get_info()[0]
    assert plan.info()["dense_windows"] == 0
    assert used <= (15 if fp8 else 18) * M * n


def test_e4m3_plan_wide_sddmm_takes_whole_tiles(gb):
    """4.4% of entries, most in full 16 x 8 blocks: at Kd = 512 whole tiles pay, at 256 they do not."""
    import torch

    M, K = 4096, 4096
    g = torch.Generator("cuda").manual_seed(777)
    at = torch.randperm(M // 16 * (K // 8), device="cuda", generator=g)[:5500]
    mask = torch.rand(M // 16, 16, K // 8, 8, device="cuda", generator=g) < 0.002
    mask[at // (K // 8), :, at % (K // 8), :] = True
    row, col = mask.view(M, K).nonzero(as_tuple=True)
    rp = torch.zeros(M + 1, dtype=torch.int32, device="cuda")
    rp[1:] = mask.view(M, K).sum(1).cumsum(0).int()
    v = torch.ones(row.numel(), device="cuda")
    plan = gb.TcPlan(rp, col.int(), v.to(torch.float8_e4m3fn).view(torch.uint8), K, row_scale=torch.ones(M, device="cuda"))
    one = torch.ones(K, device="cuda")
    for Kd, whole in ((256, False), (512, True)):
        X, Y = gen.dense_int(M, Kd, 778, -4, 4), gen.dense_int(K, Kd, 779, -4, 4)
        out, n = launches(gb, lambda: plan.sddmm(v, dev(oracle.e4m3_round(X)), dev(oracle.e4m3_round(Y)), x_scale=one, y_scale=one))
        plan.check()
        assert (n == 1) == whole
        assert torch.equal(out.double(), (dev(X).double()[row] * dev(Y).double()[col]).sum(1))


@pytest.mark.parametrize("blocks,whole", [(1000, False), (4000, True)])
def test_dense_sddmm_is_as_exact_as_the_blocks(gb, blocks, whole):
    """5% of entries anywhere and full 16 x 8 blocks: whole tiles are the more exact ones only where the blocks
    hold a fair share (a seventh) of the entries, else the residual's CSR kernel has most of them."""
    import torch

    M, K, Kd = 8192, 4096, 256
    g = torch.Generator("cuda").manual_seed(775)
    mask = torch.rand(M, K, device="cuda", generator=g) < 0.05
    at = torch.randperm(M // 16 * (K // 8), device="cuda", generator=g)[:blocks]
    mask.view(M // 16, 16, K // 8, 8)[at // (K // 8), :, at % (K // 8), :] = True
    row, col = mask.nonzero(as_tuple=True)
    rp = torch.zeros(M + 1, dtype=torch.int32, device="cuda")
    rp[1:] = mask.sum(1).cumsum(0).int()
    sv = torch.rand(row.numel(), device="cuda", generator=g) * 2 - 1
    x, y = (torch.randn(n, Kd, device="cuda", generator=g).bfloat16() for n in (M, K))
    plan = gb.TcPlan(rp, col.int(), sv.bfloat16(), K)
    out, n = launches(gb, lambda: plan.sddmm(sv, x, y))
    plan.check()
    assert n == (1 if whole else 2)
    want = (x.double()[row] * y.double()[col]).sum(1) * sv.double()
    error = lambda o: float((o.double() - want).norm() / want.norm())
    assert error(out) <= error(plan.sddmm(sv, x, y, tiles=1))


def test_dense_sddmm_random_scales_and_infinities(gb):
    """E4M3 row scales on an E4M3 plan, padded leading dimensions; an infinity or NaN in an X or Y
    row reaches only that row's entries."""
    import torch

    A = matrix(2400, 2600, 770, 0.2, 0.45)
    X, Y = gen.dense_normal(2400, 256, 771), gen.dense_normal(2600, 256, 772)
    svals = gen.dense_normal(1, A.nnz, 773)[0]
    ones = torch.ones(A.nnz, device="cuda").to(torch.float8_e4m3fn).view(torch.uint8)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), ones, 2600, row_scale=torch.ones(2400, device="cuda"))
    qx, sx = gb.quantize_e4m3_rows(dev(X))
    qy, sy = gb.quantize_e4m3_rows(dev(Y))
    wide = torch.zeros((2600, 272), dtype=torch.uint8, device="cuda")
    wide[:, :256] = qy
    out, n = launches(gb, lambda: plan.sddmm(dev(svals), qx, wide[:, :256], x_scale=sx, y_scale=sy))
    plan.check()
    dec = lambda q, s: q.view(torch.float8_e4m3fn).float().cpu().numpy().astype(np.float64) * s.cpu().numpy()[:, None]
    ref, sc = oracle.sddmm(A.rowptr, A.colidx, svals, dec(qx, sx), dec(qy, sy))
    assert n == 1
    assert_within(out.cpu().numpy(), ref, sc, TOL32, "e4m3")
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(A.vals), 2600)
    want = plan.sddmm(dev(svals), bf16(X), bf16(Y)).cpu().numpy()
    X[130, 7], Y[700, 200] = np.nan, np.inf
    out = plan.sddmm(dev(svals), bf16(X), bf16(Y)).cpu().numpy()
    rows = np.repeat(np.arange(A.M), np.diff(A.rowptr))
    hit = (rows == 130) | (A.colidx == 700)
    assert hit.any() and np.array_equal(~np.isfinite(out), hit)
    assert np.array_equal(out[~hit], want[~hit])


def test_dense_sddmm_bounded_wait_reports_timeout(gb):
    A = matrix(2048, 2048, 780, 0.2, 0.45)
    X, Y = gen.dense_int(2048, 64, 781, -4, 4), gen.dense_int(2048, 64, 782, -4, 4)
    svals = gen.vals_int(A.nnz, 783)
    plan = gb.TcPlan(dev(A.rowptr), dev(A.colidx), bf16(A.vals), 2048)
    plan.test_withhold(2)
    plan.sddmm(dev(svals), bf16(X), bf16(Y))
    with pytest.raises(gb.GbspError, match="TIMEOUT"):
        plan.check()
    plan.test_withhold(-1)
    out = plan.sddmm(dev(svals), bf16(X), bf16(Y)).cpu().numpy()
    plan.check()
    assert np.array_equal(out.astype(np.float64), oracle.sddmm(A.rowptr, A.colidx, svals, X, Y)[0])


@pytest.mark.parametrize("Kd", [128, 208, 256])
def test_dense_sddmm_without_a_plan_any_column_order(gb, Kd):
    """AUTO on E4M3 X and Y: the row statistics, the regrouping, the tiles and the marked rows; rows with
    repeated or unordered columns go to the CUDA cores with their block."""
    import torch

    M, K = 10001, 2304
    A = matrix(M, K, 790, 0.2, 0.35)
    ci = A.colidx.copy()
    for r in (1, 700, 701):
        ci[A.rowptr[r]:A.rowptr[r + 1]] = ci[A.rowptr[r]:A.rowptr[r + 1]][::-1]
    ci[A.rowptr[10000]] = ci[A.rowptr[10000] + 1]
    svals = gen.vals_int(A.nnz, 791)
    X, Y = gen.dense_int(M, Kd, 792), gen.dense_int(K, Kd, 793)
    one = lambda n: torch.ones(n, device="cuda")
    args = dev(A.rowptr), dev(ci), dev(svals), dev(oracle.e4m3_round(X)), dev(oracle.e4m3_round(Y))
    out, n = launches(gb, lambda: gb.sddmm(*args, x_scale=one(M), y_scale=one(K)))
    want, _ = oracle.sddmm(A.rowptr, ci, svals, X, Y)
    assert n == 4 and np.array_equal(out.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("Kd", [128, 208, 256])
def test_dense_sddmm_scales_and_value_round_once(gb, Kd):
    """E4M3 with whole-number dots (exact): value times dot times both scales is within half a unit in
    the last place, 2^-24 relative, and terms of 2^-47 of the exact product."""
    import torch

    M, K = 10001, 2304
    A = matrix(M, K, 795, 0.2, 0.35)
    svals = gen.dense_normal(1, A.nnz, 796)[0]
    X, Y = gen.dense_int(M, Kd, 797), gen.dense_int(K, Kd, 798)
    sx = torch.rand(M, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) + 0.5
    sy = torch.rand(K, device="cuda", generator=torch.Generator("cuda").manual_seed(2)) + 0.5
    args = dev(A.rowptr), dev(A.colidx), dev(svals), dev(oracle.e4m3_round(X)), dev(oracle.e4m3_round(Y))
    out, n = launches(gb, lambda: gb.sddmm(*args, x_scale=sx, y_scale=sy))
    f64 = lambda s: s.cpu().numpy().astype(np.float64)
    dots, _ = oracle.sddmm(A.rowptr, A.colidx, np.ones(A.nnz), X, Y)
    want = dots * svals * np.repeat(f64(sx), np.diff(A.rowptr)) * f64(sy)[A.colidx]
    assert n == 4
    assert np.all(np.abs(f64(out) - want) <= 2.0**-24 * (1 + 1e-6) * np.abs(want))


def test_dense_sddmm_scratch_past_the_pool_is_counted(gb):
    """300 million entries need 2.4 GB of scratch, most of which the pool gives back after each call: at Kd = 128
    the row split is then the faster one (the statistics and one launch)."""
    import torch

    M, K, n = 65536, 49152, 4577
    ci = (torch.arange(n, device="cuda", dtype=torch.int32) * 10 +
          (torch.arange(M, device="cuda", dtype=torch.int32) % 10)[:, None]).reshape(-1)
    rp = torch.arange(M + 1, dtype=torch.int32, device="cuda") * n
    X, Y = gen.dense_int(M, 128, 799, -4, 4), gen.dense_int(K, 128, 800, -4, 4)
    one = lambda k: torch.ones(k, device="cuda")
    out, k = launches(gb, lambda: gb.sddmm(rp, ci, one(M * n), dev(oracle.e4m3_round(X)), dev(oracle.e4m3_round(Y)),
                                           x_scale=one(M), y_scale=one(K)))
    assert k == 2
    for r in (0, 777, M - 1):
        cols = ci[r * n:(r + 1) * n].cpu().numpy()
        assert np.array_equal(out[r * n:(r + 1) * n].cpu().numpy(), Y[cols] @ X[r])
