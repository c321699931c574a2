"""Batched NLS at the sizes where the launch splits the work differently: the
group-tile pass's tile width and span, and the right-hand sides a warp grabs at
once, follow the number of right-hand sides. Every split does the same
arithmetic per right-hand side, so a batch must give the bits its parts give.
"""
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1509_09313_gb300 as lib
    return lib


# One tile per SM (64 x 152 right-hand sides) and its neighbours, a tile's
# edges, spans of several tiles, grabs of one to eight.
@pytest.mark.parametrize("nrhs", [1, 31, 33, 65, 9727, 9728, 9729, 40000, 170001])
@pytest.mark.parametrize("k,warm", [(10, False), (10, True), (50, False), (100, True)])
def test_bpp_batch_equals_its_parts(nmf, nrhs, k, warm):
    G, _ = synth.nls_batch(k, 1, seed=40 + k)
    rng = np.random.default_rng(nrhs + k)
    # Two thirds of the right-hand sides have positive solutions (the
    # all-passive group), the others mixed signs.
    X = rng.uniform(0.1, 1.0, (nrhs, k)) - (rng.random((nrhs, k)) < 0.2) * (np.arange(nrhs) % 3 == 0)[:, None]
    B = torch.from_numpy((X @ G).astype(np.float32)).cuda()
    Gd = torch.from_numpy(G).cuda()
    pin = nmf.bool_to_passive(torch.from_numpy(X > 0)).cuda() if warm else None
    group = 1   # the SIMT pass: the bits of the per-warp solves
    old = nmf.nmf_nls_bpp_get_shape(k)
    nmf.nmf_nls_bpp_set_shape(k, 8, 8, group)
    try:
        whole = nmf.nmf_nls_bpp(Gd, B, pin)
        cuts = sorted({0, min(nrhs, 500), nrhs // 3, nrhs})
        for a, b in zip(cuts[:-1], cuts[1:]):
            part = nmf.nmf_nls_bpp(Gd, B[a:b].contiguous(),
                                   None if pin is None else pin[a:b].contiguous())
            for name in ("X", "passive", "rounds", "status"):
                assert torch.equal(part[name], whole[name][a:b]), (name, a, b)
    finally:
        nmf.nmf_nls_bpp_set_shape(k, *old)


# F below and above the L2 cache (two kernels), even and odd k (pairs of columns
# or single ones), empty rows, a row longer than a 32-entry block: each output
# row against FP64, within the FP32 sum's error.
@pytest.mark.parametrize("k", [2, 33, 50, 65, 128])
@pytest.mark.parametrize("cols", [5000, 40_000_000])
def test_spmm_small_and_streamed_factors(nmf, cols, k):
    cols = 5000 if cols == 5000 else 150_000_000 // (4 * k) + 1
    rng = np.random.default_rng(cols % 1000 + k)
    count = rng.integers(0, 25, 3001)
    count[[0, 7, 8, 3000]] = 0
    count[100] = 333
    rowptr = np.concatenate([[0], np.cumsum(count)])
    colidx = np.sort(rng.integers(0, cols, rowptr[-1])).astype(np.int32)
    rng.shuffle(colidx)
    vals = rng.uniform(-1, 1, rowptr[-1]).astype(np.float32)
    F = torch.rand((cols, k), device="cuda", generator=torch.Generator("cuda").manual_seed(k))
    rp, ci, va = (torch.from_numpy(x).cuda() for x in (rowptr.astype(np.int64), colidx, vals))
    out = nmf.nmf_mm_csr(rp, ci, va, cols, F)
    row = torch.repeat_interleave(torch.arange(3001, device="cuda"), rp.diff())
    terms = va.double()[:, None] * F[ci.long()].double()
    ref = torch.zeros((3001, k), dtype=torch.float64, device="cuda").index_add_(0, row, terms)
    size = torch.zeros_like(ref).index_add_(0, row, terms.abs())
    # n sequential FMAs: at most n roundings of the running sum.
    n = rp.diff().clamp_min(1).double()[:, None]
    assert ((out.double() - ref).abs() <= n * 2.0 ** -24 * size).all()


# The tensor-core group pass against the per-warp solves: parts of a 32-row
# quarter and a 128-row tile, more tiles than SMs, rows whose stores are not
# 16-byte aligned (k = 65, 111), first tests at and next to their bound, zero,
# non-finite and far-scaled rows, and scales at which quotients decide.
@pytest.mark.parametrize("nrhs", [1, 33, 300, 152 * 128 + 97])
@pytest.mark.parametrize("k,scale,warm", [(4, 0, False), (65, 0, False), (96, 45, False),
                                          (111, 0, True), (112, 0, False)])
def test_bpp_tensor_group_edges(nmf, nrhs, k, scale, warm):
    rng = np.random.default_rng(nrhs + k)
    f4 = np.float32
    d = np.exp2(scale * (np.arange(k) % 2 * 2 - 1)).astype(f4)
    # An M-matrix: a right-hand side >= 0 has a solution >= 0, whichever
    # entries the first test takes; the rounds tell what it took.
    G = (np.eye(k) - 0.25 * (np.eye(k, k=1) + np.eye(k, k=-1))) * d[:, None] * d
    B = (rng.uniform(0.1, 1.0, (nrhs, k)) * d).astype(f4)
    kind = np.where(np.arange(nrhs) // 32 % 2 == 1, rng.integers(0, 10, nrhs), 0)
    kind[-1] = 1
    at = rng.integers(0, k, nrhs)
    for j in range(nrhs):
        i = at[j]
        if 1 <= kind[j] <= 3:
            rest = (np.arange(k) != i)
            gmax = (np.abs(B[j]) / d)[rest].max()
            bound = f4(f4(2.0 ** -20) * gmax) * d[i]
            B[j, i] = [bound, np.nextafter(bound, f4(np.inf)), np.nextafter(bound, f4(0))][kind[j] - 1]
        elif kind[j] == 4:
            B[j] = 0
        elif kind[j] == 5:
            B[j, i] = np.nan if j % 2 else np.inf
        elif kind[j] in (6, 7):
            B[j] *= f4(2.0 ** ((-70 if kind[j] == 6 else 70) if scale == 0 else 0))
        elif kind[j] == 8:
            B[j, i] = -B[j, i]
    Gd, Bd = torch.from_numpy(G.astype(np.float64)).cuda(), torch.from_numpy(B).cuda()
    pin = nmf.bool_to_passive(torch.ones(nrhs, k, dtype=torch.bool)).cuda() if warm else None
    old = nmf.nmf_nls_bpp_get_shape(k)
    out = []
    try:
        for group in (0, 2):
            nmf.nmf_nls_bpp_set_shape(k, 8, 8, group)
            out.append(nmf.nmf_nls_bpp(Gd, Bd, pin))
    finally:
        nmf.nmf_nls_bpp_set_shape(k, *old)
    for name in ("passive", "rounds", "status"):
        assert torch.equal(out[0][name], out[1][name]), name
    ok = (out[0]["status"] == 0).cpu()
    assert torch.equal(ok, torch.from_numpy(kind != 5))
    x0, x2 = (o["X"].double().cpu()[ok] * torch.from_numpy(d).double() for o in out)
    # Rows of |G| sum to 1.5 in these scales and rows of its inverse to 2 at
    # most: the residual's accumulations (five per 16 columns, truncated to
    # 2^-23, and a dozen roundings on either side) reach x three times over.
    tol = 3 * (5 * -(-k // 16) + 16) * 2.0 ** -23
    assert ((x0 - x2).abs() <= tol * x0.abs().amax(1, keepdim=True)).all()


# The tensor-core pass with the objective, its last wave shared out: the
# residual warps are the last to release a stage of the ring, which the next
# copies overwrite at once. The same run must give the same bits every time.
@pytest.mark.parametrize("m,n,k", [(4000, 2000, 50), (2500, 3100, 20)])
def test_objective_pass_repeats_bitwise(nmf, m, n, k):
    A = torch.from_numpy(synth.dense_planted(m, n, k, 0.05)).cuda()
    W0, Ht0 = (torch.from_numpy(x).cuda() for x in synth.init_factors(m, n, k))
    first = None
    for _ in range(100):
        h = nmf.nmf_init(A, W0.clone(), Ht0.clone(), precision="bf16x3", start="warm")
        h.nmf_iterate(30)
        assert h.nmf_sync() == nmf.NMF_OK
        f = list(h.nmf_objective_history())
        h.nmf_destroy()
        first = first or f
        assert f == first


# The lanes of a warp hand each other the factor and the statistics through
# shared memory: the same batch must give the same bits and counts every time,
# in systems of 1 to 32 rows.
@pytest.mark.parametrize("k", [2, 20, 33, 48, 50, 56, 64])
def test_bpp_warp_solves_repeat_bitwise(nmf, k):
    G, B = synth.nls_batch(k, 20011, seed=k)
    Gd, Bd = torch.from_numpy(G).cuda(), torch.from_numpy(B.astype(np.float32)).cuda()
    first = nmf.nmf_nls_bpp(Gd, Bd)
    for _ in range(30):
        again = nmf.nmf_nls_bpp(Gd, Bd)
        for name in ("X", "passive", "rounds", "status"):
            assert torch.equal(first[name], again[name]), name


# Device memory the tensor-core products take beside their operands. A handle's
# scratch for a shared last wave is bounded (71 row tiles, all shared: an eighth of
# A's bytes otherwise), and nmf_mm_dense, which forms no objective, has none of it.
def test_shared_wave_scratch_is_bounded(nmf):
    m, n, k = 9000, 320000, 33
    A = torch.zeros((m, n), device="cuda")
    W0, Ht0 = torch.rand((m, k), device="cuda"), torch.rand((n, k), device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = nmf.nmf_init(A, W0, Ht0, precision="bf16x3", split_copies=False)
    used = before - torch.cuda.mem_get_info()[0]
    h.nmf_destroy()
    # Factors, right-hand sides and passive sets, both factors in BF16 halves
    # (64 columns), the Gram's and the splits' partial sums, rounded up freely.
    assert used <= 4 * (8 * (m + n) * k + 4 * (m + n) * 64) + (512 << 20), used


def used_memory(call):
    """Most bytes the device's default stream-ordered pool gave out during the call."""
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    pool, high = ctypes.c_void_p(), ctypes.c_uint64(0)
    USED_MEM_HIGH = 8
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    call()
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert high.value > 0
    return high.value


def test_mm_dense_takes_no_objective_scratch(nmf):
    m, n, k = 9728, 16000, 50
    A, F = torch.rand((m, n), device="cuda"), torch.rand((n, k), device="cuda")
    used = used_memory(lambda: nmf.nmf_mm_dense(A, F, False, "bf16x3"))
    # F in BF16 halves and at most four partial sums of the output.
    assert used <= 4 * n * 64 + 4 * 4 * m * k + (1 << 20), used


# One call maps the scratch of a shared last wave afresh: it is taken only where
# it pays (76 tiles are half a wave; 36 of 24 columns, 18 narrow ones beside a whole
# wave). F^T, the output and, of the objective, both factors' halves remain.
@pytest.mark.parametrize("m,k", [(9728, 50), (4608, 24), (21760, 10)])
def test_one_call_takes_no_scratch_that_does_not_pay(nmf, m, k):
    n = 16000
    A, F = torch.rand((m, n), device="cuda"), torch.rand((n, k), device="cuda")
    W = torch.rand((m, k), device="cuda")
    few = 4 * n * 64 + 4 * m * k + (1 << 20)
    used = used_memory(lambda: nmf.nmf_mm_dense(A, F, False, "fp32"))
    assert used <= few, used
    if k == 50:
        used = used_memory(lambda: nmf.nmf_objective_dense(A, W, F, "bf16x3"))
        assert used <= few + 4 * m * 64, used


# The same shapes unshared against their parts shared: the products to the bit; the
# objective, whose residuals are the same but summed in other groups (compensated FP32
# sums per thread, FP64 across), to the rounding of those sums.
@pytest.mark.parametrize("m,k", [(9728, 50), (4608, 24), (21760, 10)])
def test_unshared_and_shared_waves_agree(nmf, m, k):
    n = 16000
    g = torch.Generator("cuda").manual_seed(m)
    A, F = (torch.rand(s, device="cuda", generator=g) for s in ((m, n), (n, k)))
    W = torch.rand((m, k), device="cuda", generator=g)
    whole = nmf.nmf_mm_dense(A, F, False, "fp32")
    f = nmf.nmf_objective_dense(A, W, F, "bf16x3")
    parts = 0.0
    for a in range(0, m, 2304):   # 18 tiles and what is left
        b = min(m, a + 2304)
        assert torch.equal(nmf.nmf_mm_dense(A[a:b], F, False, "fp32"), whole[a:b]), a
        parts += nmf.nmf_objective_dense(A[a:b], W[a:b], F, "bf16x3")
    assert abs(parts - f) <= 2.0 ** -22 * f


# A H^T in FP32 with the last wave's tiles shared out, alone or behind a whole wave
# (152 tiles of 128 rows), against the same rows multiplied alone or unshared: a
# row's sums do not depend on the grid, to the bit. Column chunks of every width,
# two chunks (k = 100), a contraction that ends inside a stage; 38 tiles are shared
# by four CTAs each, 18 by eight, 77 by none.
@pytest.mark.parametrize("k", [10, 24, 40, 50, 64, 100])
def test_mm_fp32_rows_do_not_depend_on_the_grid(nmf, k):
    n = 2003 + 1
    g = torch.Generator("cuda").manual_seed(k)
    A = torch.rand((170 * 128 + 5, n), device="cuda", generator=g) - 0.3
    F = torch.rand((2003, k), device="cuda", generator=g) - 0.3
    A = A[:, :2003]
    whole = nmf.nmf_mm_dense(A, F, False, "fp32")
    for a, b in ((0, 38 * 128), (0, 18 * 128), (152 * 128, 170 * 128 + 5), (0, 77 * 128), (128, 129)):
        assert torch.equal(nmf.nmf_mm_dense(A[a:b], F, False, "fp32"), whole[a:b]), (a, b)


# Long rows side by side (a matrix sorted by degree) in the streamed product: they
# are dealt out to the warps row by row, at the edges of stretches of 16 rows and
# of 2, and at the last, cut-off stretch. A row's sum does not depend on where the
# row stands, to the bit, and lies within the FP32 sum's error of the FP64 one.
@pytest.mark.parametrize("rows", [19463, 160001])
@pytest.mark.parametrize("k", [33, 50, 100])
def test_spmm_long_rows_side_by_side(nmf, rows, k):
    cols = 150_000_000 // (4 * k) + 1
    rng = np.random.default_rng(rows + k)
    count = rng.integers(0, 4, rows)
    count[4001:4107] = 3000
    count[8007] = 40001
    count[rows - 3:] = [2500, 0, 2500]
    count[0], count[16] = 2049, 2047
    ptr = np.concatenate([[0], np.cumsum(count)]).astype(np.int64)
    col = rng.integers(0, cols, ptr[-1]).astype(np.int32)
    val = rng.uniform(-1, 1, ptr[-1]).astype(np.float32)
    F = torch.rand((cols, k), device="cuda", generator=torch.Generator("cuda").manual_seed(k))

    def product(order):
        at = np.concatenate([np.arange(ptr[r], ptr[r + 1]) for r in order])
        p = np.concatenate([[0], np.cumsum(count[order])]).astype(np.int64)
        return nmf.nmf_mm_csr(*(torch.from_numpy(x).cuda() for x in (p, col[at], val[at])), cols, F)

    out = product(np.arange(rows))
    order = rng.permutation(rows)
    assert torch.equal(product(order), out[torch.from_numpy(order).cuda()])
    for r in (0, 16, 4001, 4106, 8007, rows - 3, rows - 2, rows - 1, 5000):
        e = slice(int(ptr[r]), int(ptr[r + 1]))
        terms = (torch.from_numpy(val[e]).cuda().double()[:, None]
                 * F[torch.from_numpy(col[e]).cuda().long()].double())
        # n sequential FMAs: at most n roundings of the running sum.
        assert ((out[r].double() - terms.sum(0)).abs()
                <= max(count[r], 1) * 2.0 ** -24 * terms.abs().sum(0)).all(), r


# Partial sums of a split contraction are added in FP64 and rounded once (A H^T in
# FP32 has one chain and none). Three terms in three splits: 1 + 2^-24 lies in the
# middle of two floats, and 2^-50 decides; further on sums that cancel, that overflow
# FP32 on the way and that end subnormal.
@pytest.mark.parametrize("precision,trans", [("fp32", True), ("bf16x3", True), ("bf16x3", False)])
def test_split_sums_round_once(nmf, precision, trans):
    Q, P, k = 16000, 128, 8
    h = 2.0 ** -24
    terms = [(1, h, 2.0 ** -50), (1, h, -(2.0 ** -50)), (1, 2 * h, -(2.0 ** -50)),
             (1, 0, -(2.0 ** -50)), (-1, -h, -(2.0 ** -50)), (h, 2.0 ** -50, 1),
             (2.0 ** -50, 1, h), (3 * h, 1, 2.0 ** -60), (1 + 2.0 ** -6, -1, 2.0 ** -70), (0, 0, 0)]
    if precision == "fp32":
        terms += [(2.0 ** 127, 2.0 ** 127, -(2.0 ** 127)),
                  (1.5 * 2.0 ** -130, 2.0 ** -140, -(2.0 ** -133))]
    A = torch.zeros((P, Q))
    at = [0, Q // 2, Q - 1]
    for r, t in enumerate(terms):
        A[r, at] = torch.tensor(t, dtype=torch.float32)
    want = [np.float32(np.float64(np.float64(a) + np.float64(b)) + np.float64(c))
            for a, b, c in terms]
    Ad = (A.T.contiguous() if trans else A).cuda()
    out = nmf.nmf_mm_dense(Ad, torch.ones((Q, k), device="cuda"), trans, precision).cpu().numpy()
    for r, w in enumerate(want):
        assert np.array_equal(out[r], np.full(k, w, np.float32)), (r, out[r], w)
