"""Sizes at the edges of the kernels' tiles, chunks and rounds, against the oracle.

Every size here sits on one side or the other of a tile, a K tile, a round of
reconstructed bins, a chunk of constants or a dispatch threshold."""

import numpy as np
import pytest

import oracle as O
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def srw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_00488_gb300 as pkg
    return pkg


def line_workload(n_t, n_rec, exposure=2.0e4):
    """One 7Be line on [0, 1] MeV with a few empty-data bins at the top."""
    t_edges, rec_edges = np.linspace(0.0, 1.0, n_t + 1), np.linspace(0.0, 1.3, n_rec + 1)
    r = workloads.solar.response_matrix(t_edges, rec_edges, res=0.06, tail_frac=1e-3)
    return {"name": "line", "t_edges": t_edges, "rec_edges": rec_edges, "sources": workloads.solar.be7_sources(), "R": r,
            "bkg": np.full((1, n_rec), 0.1 * exposure / n_rec), "exposure": exposure, "t_min": 1e-3, "sin2w": 0.23121,
            "f_tau": 0.5}


def model_and_counts(wl, mask=None):
    m = O.OracleModel.from_workload(wl)
    m.set_data(np.zeros(wl["R"].shape[0]), wl["bkg"])
    counts = workloads.poisson_counts(m.mu(np.zeros(5)), 3)
    m.set_data(counts, wl["bkg"], mask)
    return m, counts


def oracle_matrix(m):
    """The folded signal per coupling monomial, [8, n_rec] (FP64): many points without many spectra."""
    basis = O.coefficient_spectra(m.sources, m.t_edges, m.t_min)
    safe = np.where(m.s_sm != 0, m.s_sm, 1.0)
    shat = np.where(m.s_sm != 0, basis * (m.e_sm / safe), 0.0)
    shat[6] = np.where(m.s_sm != 0, shat[6], m.e_sm)
    return shat @ m.r.T


def values(m, M, theta):
    from scipy.special import gammaln, xlogy
    c = np.array([O.coupling_coefficients(t) for t in theta.astype(np.float64)])
    mu = c @ M + m.bkg_sum
    t = 2.0 * (mu - xlogy(m.counts, mu) + gammaln(m.counts + 1.0))
    return (t * (1.0 if m.mask is None else (m.mask != 0))).sum(1), mu


# FP32 products: |d(-2 ln L)| <= 1e-4 in the fit region (the library's bar)
@pytest.mark.parametrize("n_t,n_rec,p", [(1, 1, 2), (15, 63, 31), (16, 64, 33), (17, 65, 64), (65, 127, 65), (64, 129, 2),
                                         (260, 385, 700), (100, 2050, 640)])
def test_fp32_batch_tiles(srw, n_t, n_rec, p):
    wl = line_workload(n_t, n_rec)
    mask = (np.arange(n_rec) % 7 != 3).astype(np.uint8) if n_rec > 1 else None
    m, counts = model_and_counts(wl, mask)
    theta = workloads.fit_region_points(p, seed=n_rec)
    want, mu = values(m, oracle_matrix(m), theta)
    with srw.Likelihood(wl, counts, mask=mask) as lk:
        got = lk.loglik(theta, srw.SRW_FP32)
        spec = lk.spectrum_batch(theta, srw.SRW_FP32)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-4)
    np.testing.assert_allclose(spec, mu - m.bkg_sum, rtol=1e-6, atol=1e-6 * mu.max())


# rank 8: every path adds the same terms in the same order, so a point's value,
# gradient and profiled value do not depend on the size of the batch that holds
# it, which decides the path.  (The oracle's values: test_gpu_parity.py.)
@pytest.mark.parametrize("n_rec,p", [(1, 16), (63, 17), (64, 2432), (65, 2433), (129, 4865), (1025, 33), (2049, 40),
                                     (70, 9728), (70, 19455), (257, 19456)])
def test_rank8_and_profiled_rounds(srw, n_rec, p):
    wl = line_workload(50, n_rec)
    mask = (np.arange(n_rec) % 5 != 2).astype(np.uint8) if n_rec > 1 else None
    _, counts = model_and_counts(wl, mask)
    theta = workloads.fit_region_points(p, seed=p)
    with srw.Likelihood(wl, counts, mask=mask) as lk:
        v, g = lk.loglik_linear(theta, grad=True)
        only = lk.loglik_linear(theta)
        prof, alpha = lk.loglik_profiled(theta[:5000], 0.05)
        assert np.all(np.isfinite(v)) and np.all(np.isfinite(g)) and np.all(np.isfinite(prof))
        np.testing.assert_array_equal(only, v)
        for k in (0, p // 2, p - 1):
            v1, g1 = lk.loglik_linear(theta[k:k + 1], grad=True)
            assert v1[0] == v[k] and np.array_equal(g1[0], g[k])
            if k < len(prof):
                p1, a1 = lk.loglik_profiled(theta[k:k + 1], 0.05)
                assert p1[0] == prof[k] and a1[0] == alpha[k]


# The single-point spectrum sums up to 128 nodes in the bins' blocks, more in
# chunks of 32 (longer ones from 8193 nodes on), and the bins 32 to a block; some bins lie below the threshold, some
# hold many clipped nodes, the topmost none.  S is an FP64 sum rounded to FP32
# (6e-8); its terms cancel to (m_e / (m_e + 2E))^2 >= 2e-4, so 1e-7 holds with
# room for the FP64 rounding of up to 2e4 terms.
@pytest.mark.parametrize("midpoint", [False, True])
@pytest.mark.parametrize("n_nodes,n_t", [(1, 1), (31, 33), (32, 32), (33, 31), (128, 7), (129, 7), (1000, 5), (8192, 64),
                                         (8193, 257), (20000, 100)])
def test_spectrum_node_chunks_and_bin_blocks(srw, n_nodes, n_t, midpoint):
    rng = np.random.default_rng(n_nodes + n_t)
    e = rng.uniform(0.2, 16.0, n_nodes)
    src = [{"name": "s", "e": e, "w": rng.uniform(0.1, 1.0, n_nodes), "pee": rng.uniform(0.3, 0.6, n_nodes)}]
    t_edges = np.linspace(0.0, 17.0, n_t + 1)
    wl = line_workload(n_t, 8)
    wl.update(sources=src, t_edges=t_edges, t_min=0.3 if n_t > 1 else 1e-3)
    theta = np.array([[0.11, -0.07, 0.21, 0.05, 1.3], [0.0, 0.0, 0.0, 0.0, 0.0]], np.float32)
    with srw.Likelihood(wl, midpoint=midpoint, e_true_sm=np.ones(n_t)) as lk:  # one centre above T_max: S_SM = 0
        for t in theta:
            want = O.recoil_spectrum(src, t_edges, t.astype(np.float64), wl["t_min"], wl["sin2w"], wl["f_tau"],
                                     midpoint=midpoint)
            got = lk.spectrum(t, 0)
            np.testing.assert_allclose(got, want, rtol=1e-7, atol=0)
            np.testing.assert_array_equal(got == 0, want == 0)


# Tensor-core fold: per (rec tile, block of 64 true bins) only the rows of R with
# nonzero split elements are multiplied.  Bands that start and end anywhere,
# single elements at a block's corners, empty rows and an empty tile.  Bound:
# the dropped lo x lo product and the splits' residuals (2^-15 / 2^-21 of each
# product of R with W - W_ref), FP32 accumulation over n_t terms, one rounding
# of the result and of the FP32 spectra.
@pytest.mark.parametrize("prec,split", [("bf16x3", 2.0**-15), ("fp16x3", 2.0**-21)])
@pytest.mark.parametrize("n_t,n_rec,form", [(300, 300, "band"), (65, 257, "corners"), (257, 520, "gap"), (129, 16, "band")])
def test_tensor_fold_rows_left_out(srw, n_t, n_rec, form, prec, split):
    wl = line_workload(n_t, n_rec)
    r = wl["R"].copy()
    i, j = np.arange(n_t)[None, :], np.arange(n_rec)[:, None]
    if form == "band":
        keep = np.abs(i / n_t - j / n_rec - 0.07) < 0.06
    elif form == "corners":
        keep = ((i % 64 == 0) | (i % 64 == 63) | (i == n_t - 1)) & ((j % 16 == 0) | (j % 16 == 15) | (j == n_rec - 1))
        r = np.maximum(r, 1e-6)
    else:
        keep = (j < 250) | (j >= 513)  # rows 256..511, a whole tile, are empty
    wl["R"] = np.ascontiguousarray(np.where(keep, r, 0.0), dtype=r.dtype)
    m, counts = model_and_counts(wl)
    theta = workloads.fit_region_points(130, seed=n_t)
    basis = O.coefficient_spectra(m.sources, m.t_edges, m.t_min)
    shat = np.where(m.s_sm != 0, basis * (m.e_sm / np.where(m.s_sm != 0, m.s_sm, 1.0)), 0.0)
    c = np.array([O.coupling_coefficients(t) for t in theta.astype(np.float64)])
    dw = (c - O.coupling_coefficients(np.zeros(5))) @ shat
    _, mu = values(m, oracle_matrix(m), theta)
    bound = (split + n_t * 2.0**-24) * (np.abs(dw) @ m.r.T) + 2.0**-22 * mu
    with srw.Likelihood(wl, counts) as lk:
        spec = lk.spectrum_batch(theta, srw.PRECISIONS[prec])
    assert np.all(np.abs(spec - (mu - m.bkg_sum)) <= bound)


# Surrogate: the scan takes 256 points a unit and the GEMM tiles narrow for few
# rows; every output adds the same products in the same order, so a point's
# outputs and value do not depend on the size of the batch that holds it.
@pytest.mark.parametrize("n_rec", [1, 255, 257, 600])
def test_surrogate_batch_sizes(srw, n_rec):
    from workloads.mlp import BOX_CENTRE, BOX_HALF, init_weights, round_to_bf16
    wl = line_workload(64, n_rec)
    _, counts = model_and_counts(wl)
    params = [(round_to_bf16(W), round_to_bf16(b)) for W, b in init_weights(n_rec, seed=5)]
    theta = workloads.theta_box(40000, 43)
    with srw.Likelihood(wl, counts) as lk:
        s = srw.Surrogate(lk, params, BOX_CENTRE, BOX_HALF)
        try:
            y, v = s.forward(theta[:20000]), s.loglik(theta)
            assert np.all(np.isfinite(v))
            for p in (1, 127, 129, 255, 256, 257, 4096):
                np.testing.assert_array_equal(s.forward(theta[:p]), y[:p])
                np.testing.assert_array_equal(s.loglik(theta[:p]), v[:p])
        finally:
            s.close()
