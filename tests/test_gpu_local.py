"""MU (Eq. 5) and HALS (Eq. 6) on the GPU against the FP64 oracle.

One step of either update is a fixed function of (G, R, X); the kernels work
in FP32 (G rounded to FP32, products accumulated in FP32), so an entry carries
an error of a few units of FP32 rounding times the size of the terms it sums:
MU ~ k * 6e-8 relative, HALS a little more (each coordinate uses the others'
new values). The tolerances below are 2e-5 of each row's scale. Whole ANLS
runs compare the objective history (1e-5 relative, as for BPP) and the
factors (1e-4 relative Frobenius).
"""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1509_09313_gb300 as lib
    return lib


def dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda()


def problem(rows, k, seed, zero_frac=0.2):
    rng = np.random.default_rng(seed)
    C = rng.uniform(0.0, 1.0, (4 * k + 8, k))
    G = C.T @ C
    X = rng.uniform(0.0, 1.0, (rows, k)) * (rng.uniform(0, 1, (rows, k)) > zero_frac)
    R = rng.uniform(0.0, 1.0, (rows, k)) @ G * 0.8
    return G, R.astype(np.float32), X.astype(np.float32)


def row_rel_err(got, ref):
    scale = np.maximum(np.abs(ref).max(axis=1, keepdims=True), 1e-30)
    return float((np.abs(got - ref) / scale).max())


@pytest.mark.parametrize("k", [1, 7, 32, 33, 50, 64, 65, 100, 128])
@pytest.mark.parametrize("solver", ["mu", "hals"])
def test_step_matches_oracle(nmf, solver, k):
    rows = 1000 + 37   # several CTAs, a ragged last one
    G, R, X = problem(rows, k, seed=k)
    Xd = dev(X)
    fn = nmf.nmf_update_mu if solver == "mu" else nmf.nmf_update_hals
    fn(dev(G, torch.float64), dev(R), Xd)
    got = Xd.double().cpu().numpy()
    ref = (oracle.mu if solver == "mu" else oracle.hals)(G, R, X)
    err = row_rel_err(got, ref)
    print(f"{solver} k={k} max row-relative error {err:.2e}")
    assert err <= 2e-5, err
    assert (got >= 0).all()


def test_mu_zero_rows_and_hals_zero_column(nmf):
    k, rows = 12, 300
    G, R, X = problem(rows, k, seed=3)
    X[::5] = 0.0                       # MU: (X G) = 0 on these rows; they stay 0
    Xd = dev(X)
    nmf.nmf_update_mu(dev(G, torch.float64), dev(R), Xd)
    got = Xd.cpu().numpy()
    assert np.isfinite(got).all() and (got[::5] == 0).all()
    G0 = G.copy()
    G0[4, :] = 0.0
    G0[:, 4] = 0.0                     # HALS: G_44 = 0 sets x_4 to 0
    Xd = dev(X + 1.0)
    nmf.nmf_update_hals(dev(G0, torch.float64), dev(R), Xd)
    got = Xd.double().cpu().numpy()
    assert (got[:, 4] == 0).all()
    ref = oracle.hals(G0, R, X + 1.0)
    assert row_rel_err(got, ref) <= 2e-5


def test_empty_batch_is_a_no_op(nmf):
    G = dev(np.eye(5), torch.float64)
    X = torch.empty((0, 5), dtype=torch.float32, device="cuda")
    R = torch.empty((0, 5), dtype=torch.float32, device="cuda")
    nmf.nmf_update_mu(G, R, X)
    nmf.nmf_update_hals(G, R, X)
    torch.cuda.synchronize()


def run_anls(nmf, A, W0, Ht0, iters, solver, precision="fp32", csr=None, shape=None):
    Ad = dev(A) if csr is None else tuple(torch.from_numpy(x).cuda() for x in csr)
    h = nmf.nmf_init(Ad, dev(W0), dev(Ht0), precision=precision, solver=solver, shape=shape)
    h.nmf_iterate(iters)
    assert h.nmf_sync() == nmf.NMF_OK
    W, Ht = h.nmf_get_factors()
    f = np.array(h.nmf_objective_history())
    st = h.nmf_get_stats()
    h.nmf_destroy()
    assert st["bpp_rhs"] == 0          # no BPP solve ran
    return W.double().cpu().numpy(), Ht.double().cpu().numpy(), f


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
@pytest.mark.parametrize("solver", ["mu", "hals"])
def test_anls_dense_matches_oracle(nmf, solver, precision):
    m, n, k, T = 2000, 1000, 10, 10
    A = synth.dense_planted(m, n, k, 0.01)
    W0, Ht0 = synth.init_factors(m, n, k)
    ref = oracle.anls(A, W0, Ht0, iters=T, solver=solver)
    W, Ht, f = run_anls(nmf, A, W0, Ht0, T, solver, precision)
    errf = np.abs(f - ref["f"][1:]) / ref["f"][1:]
    errW = np.linalg.norm(W - ref["W"]) / np.linalg.norm(ref["W"])
    errH = np.linalg.norm(Ht - ref["Ht"]) / np.linalg.norm(ref["Ht"])
    print(f"{solver}/{precision}: f {errf.max():.2e}  W {errW:.2e}  H {errH:.2e}")
    assert errf.max() <= 1e-5
    assert errW <= 1e-4 and errH <= 1e-4
    assert (f[1:] <= f[:-1] * (1 + 1e-6)).all()   # both updates never increase f


@pytest.mark.parametrize("solver", ["mu", "hals"])
def test_anls_sparse_matches_oracle(nmf, solver):
    m, n, k, T = 20000, 10000, 20, 5
    csr = synth.csr_uniform(m, n, 200000)
    W0, Ht0 = synth.init_factors(m, n, k)
    ref = oracle.anls(None, W0, Ht0, iters=T, csr=csr, shape=(m, n), solver=solver)
    W, Ht, f = run_anls(nmf, None, W0, Ht0, T, solver, csr=csr, shape=(m, n))
    errf = np.abs(f - ref["f"][1:]) / ref["f"][1:]
    errW = np.linalg.norm(W - ref["W"]) / np.linalg.norm(ref["W"])
    errH = np.linalg.norm(Ht - ref["Ht"]) / np.linalg.norm(ref["Ht"])
    print(f"sparse {solver}: f {errf.max():.2e}  W {errW:.2e}  H {errH:.2e}")
    assert errf.max() <= 1e-5
    assert errW <= 1e-4 and errH <= 1e-4


def test_proposal_rejected_for_mu(nmf):
    m, n, k = 200, 100, 8
    A = synth.dense_planted(m, n, k, 0.01)
    W0, Ht0 = synth.init_factors(m, n, k)
    h = nmf.nmf_init(dev(A), dev(W0), dev(Ht0), solver="mu")
    net = nmf.nmf_mlp_create(k, 16, torch.from_numpy(synth.mlp_init(k, 16)).cuda())
    with pytest.raises(nmf.NMFError):
        h.nmf_set_proposal(net, "train")
    h.nmf_destroy()


# Row counts at the edges of the kernels (one warp per row, 64-row tiles from 48 or
# 384 rows per SM on, their last one ragged), block edges of k. Same bound as above.
@pytest.mark.parametrize("rows", [1, 31, 33, 7295, 7297, 38913, 58367, 58369])
@pytest.mark.parametrize("k", [1, 8, 9, 50, 64, 65, 128])
@pytest.mark.parametrize("solver", ["mu", "hals"])
def test_step_at_tile_edges(nmf, solver, k, rows):
    G, R, X = problem(rows, k, seed=rows + k)
    Xd = dev(X)
    fn = nmf.nmf_update_mu if solver == "mu" else nmf.nmf_update_hals
    fn(dev(G, torch.float64), dev(R), Xd)
    ref = (oracle.mu if solver == "mu" else oracle.hals)(G, R, X)
    assert row_rel_err(Xd.double().cpu().numpy(), ref) <= 2e-5


# MU takes tiles only where their last wave is full enough, by k and the warps that
# fit (k = 25, 40, 56, 64, 100, 112, 128 on 152 SMs): both sides of each line. Same
# bound.
@pytest.mark.parametrize("k,rows", [(25, 87488), (25, 87616), (40, 69952), (40, 70080),
                                    (56, 78144), (56, 78272), (64, 79744), (64, 79808),
                                    (100, 76992), (100, 77056), (112, 80704), (112, 80768),
                                    (128, 73920), (128, 73984), (96, 58369)])
def test_mu_at_the_lines_of_partial_waves(nmf, k, rows):
    G, R, X = problem(rows, k, seed=rows + k)
    Xd = dev(X)
    nmf.nmf_update_mu(dev(G, torch.float64), dev(R), Xd)
    assert row_rel_err(Xd.double().cpu().numpy(), oracle.mu(G, R, X)) <= 2e-5


# The division of HALS's coordinate on both sides of the switch between its two
# kernels (48 rows per SM; 152 SMs): k = 1 makes x = max(r, 0) / g of every row,
# which the FP32 division rounds to nearest. Diagonals down to the smallest
# subnormal (their reciprocals overflow) and up to 1e38, numerators of every size
# and zero and negative ones; then k = 3, where a column of such a norm stands
# beside ordinary ones and is clamped to zero.
@pytest.mark.parametrize("rows", [7295, 7297])
@pytest.mark.parametrize("g", [1e-45, 1e-41, 2.0 ** -129, 2.0 ** -128, 2.0 ** -126, 3e-38, 1.1e-30,
                               7e-20, 0.3, 1.0, 3.7e8, 9e29, 1.1e30, 2.0 ** 126, 1e38, 3.4e38])
def test_hals_quotient_is_the_rounded_one(nmf, g, rows):
    rng = np.random.default_rng(rows)
    r = (np.exp2(rng.uniform(-149, 127.9, rows)) * rng.choice([-1, 1, 1, 1], rows)).astype(np.float32)
    r[::5] = 0.0
    with np.errstate(over="ignore"):
        r[1::7] = np.float32(g) * rng.uniform(0.5, 2.0, r[1::7].shape).astype(np.float32)
    X = dev(rng.uniform(0, 1, (rows, 1)))
    nmf.nmf_update_hals(dev([[g]], torch.float64), dev(r[:, None]), X)
    with np.errstate(over="ignore"):
        want = np.maximum(r, np.float32(0)) / np.float32(g)
    assert np.array_equal(X.cpu().numpy()[:, 0], want)

    G = np.diag([4.0, g, 2.0])
    R = np.stack([rng.uniform(1, 2, rows), -rng.uniform(0, 1, rows), rng.uniform(1, 2, rows)], 1)
    X = dev(rng.uniform(0, 1, (rows, 3)))
    nmf.nmf_update_hals(dev(G, torch.float64), dev(R), X)
    R = R.astype(np.float32)
    want = np.stack([R[:, 0] / np.float32(4), np.zeros(rows, np.float32), R[:, 2] / np.float32(2)], 1)
    assert np.array_equal(X.cpu().numpy(), want)


# Infinities, NaN and sums that overflow, on both sides of the switch between the
# kernels: the same answer. A negative sum beyond the range (only a Gram with
# negative entries has one) makes the coordinate infinite, not zero.
def test_hals_special_values_in_both_kernels(nmf):
    k, rows = 5, 7297
    G = np.eye(k) * 3 + 0.5
    G[0, 3] = G[3, 0] = -2.0
    G[1, 2] = G[2, 1] = 0.0
    X = np.full((rows, k), 0.5, np.float32)
    R = np.full((rows, k), 2.0, np.float32)
    X[0::8, [0, 3]] = 3e38
    R[1::8, 1] = np.inf
    R[2::8, 1] = -np.inf
    R[3::8, 1] = np.nan
    R[4::8] = 3e38
    whole, part = dev(X), dev(X[:1000])
    nmf.nmf_update_hals(dev(G, torch.float64), dev(R), whole)
    nmf.nmf_update_hals(dev(G, torch.float64), dev(R[:1000]), part)
    a, b = whole[:1000].cpu().numpy(), part.cpu().numpy()
    assert np.isposinf(a[0::8, 0]).all() and np.isposinf(a[1::8, 1]).all()
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    assert np.array_equal(a[~np.isfinite(b)], b[~np.isfinite(b)], equal_nan=True)
    # Finite ones: the kernels' sums round differently, a few units of 2^-24.
    fin = np.isfinite(b)
    assert (np.abs(a[fin].astype(np.float64) - b[fin]) <= 16 * 2.0 ** -24 * np.abs(b[fin])).all()
