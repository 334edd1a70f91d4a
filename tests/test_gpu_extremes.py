"""Values at the ends of what the evaluators take, and in batches of other sizes.

Bins with almost no expectation beside their data, counts below FP32's range,
empty bins beside ordinary ones, batches on either side of the tile and unit
rules (a point's value may not depend on the batch that holds it), very many
reconstructed bins, and a surrogate pass whose device wait runs out.
"""

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
    pkg.srw_fault_inject("none")
    yield pkg
    pkg.srw_fault_inject("none")


def line(n_t, n_rec, exposure=2.0e4):
    """One 7Be line on [0, 1] MeV, smeared onto n_rec bins of [0, 1.3] MeV."""
    t_edges, rec_edges = np.linspace(0.0, 1.0, n_t + 1), np.linspace(0.0, 1.3, n_rec + 1)
    r = workloads.solar.response_matrix(t_edges, rec_edges, res=0.06, tail_frac=1e-3)
    return {"name": "line", "t_edges": t_edges, "rec_edges": rec_edges, "sources": workloads.solar.be7_sources(), "R": r,
            "bkg": np.full((1, n_rec), 0.1 * exposure / n_rec), "exposure": exposure, "t_min": 1e-3, "sin2w": 0.23121,
            "f_tau": 0.5}


def oracle_of(wl, counts=None):
    m = O.OracleModel.from_workload(wl)
    m.set_data(np.zeros(wl["R"].shape[0]), wl["bkg"])
    if counts is None:
        counts = workloads.poisson_counts(m.mu(np.zeros(5)), 3)
    m.set_data(counts, wl["bkg"])
    return m, counts


def with_bins(n_t, n_rec, bins):
    """The line with given expectations (no background) and counts in some bins: {bin: (mu, n)}."""
    wl = line(n_t, n_rec)
    r, bkg = wl["R"].copy(), wl["bkg"].copy()
    m, counts = oracle_of(wl)
    total = float(m.e_sm.sum())
    for j, (mu, n) in bins.items():
        r[j, :] = np.float32(mu / total)
        bkg[:, j] = 0.0
        counts[j] = n
    wl.update(R=r, bkg=bkg, e_true_sm=m.e_sm)
    return wl, counts


# A count beside an expectation of 1e-30 .. 1e-24: n / mu beyond 2^100.  FP32
# products: |d(-2 ln L)| <= 1e-4 in the fit region (the library's bar; a relative
# error of 2^-24 of the deviation from the reference moves the three terms by at
# most 2 x 3 x 1e3 x 2^-24 x 0.1 = 4e-5), and 2^-50 of the sum for its rounding.
@pytest.mark.parametrize("p", [3, 10000])
@pytest.mark.parametrize("n,mu", [(10.0, 1.1e-30), (100.0, 1.5e-30), (100.0, 1e-29), (100.0, 1e-28), (1e3, 1e-26),
                                  (1e3, 1e-24), (3.0, 1e-31)])
def test_fp32_batch_counts_without_expectation(srw, n, mu, p):
    wl, counts = with_bins(64, 130, {0: (mu, n), 70: (mu, n), 129: (mu, n)})
    m = O.OracleModel.from_workload(wl, e_true_sm=wl["e_true_sm"])
    m.set_data(counts, wl["bkg"])
    theta = workloads.fit_region_points(p, seed=7)
    pick = np.unique(np.linspace(0, p - 1, 5).astype(int))
    want = m.neg2lnl_batch(theta[pick].astype(np.float64))
    with srw.Likelihood(wl, counts, e_true_sm=wl["e_true_sm"]) as lk:
        got = lk.loglik(theta, srw.SRW_FP32)[pick]
    np.testing.assert_allclose(got, want, rtol=2.0**-50, atol=1e-4)


# FP32 products at the reference point, where the fold's deviation is exactly 0:
# what is left is the Poisson term of mu = b + R W_ref (FP64) in double-float.
# Its bound is 1.4e-13 (n + mu), twice that for -2 ln L; 2e-14 (n + mu) more for
# mu and the data constant, sums of a few hundred FP64 terms in either program.
def test_fp32_batch_poisson_term_at_the_reference(srw):
    wl = line(40, 1, exposure=3.0e3)
    m, _ = oracle_of(wl)
    mu = float(m.mu(np.zeros(5))[0])
    theta = np.zeros((2, 5), np.float32)
    worst = 0.0
    for ratio in np.concatenate([np.linspace(0.70, 0.75, 12), np.linspace(1.3, 1.42, 12), [0.01, 0.3, 1.001, 7.0, 60.0]]):
        counts = np.array([np.floor(mu * ratio) + 1.0])
        m.set_data(counts, wl["bkg"])
        with srw.Likelihood(wl, counts) as lk:
            got = lk.loglik(theta, srw.SRW_FP32)
        worst = max(worst, np.max(np.abs(got - m.neg2lnl(theta[0]))) / (counts[0] + mu))
    assert worst <= 3.0e-13


# A count below FP32's range in a bin that expects nothing: outside the domain.
@pytest.mark.parametrize("n", [1.0, 1e-40, 1e-50])
def test_fp32_batch_tiny_count_is_data(srw, n):
    wl, counts = with_bins(64, 130, {70: (0.0, n)})
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    theta = torch.from_numpy(workloads.fit_region_points(3, seed=7)).cuda()
    with srw.Likelihood(wl, counts, e_true_sm=wl["e_true_sm"]) as lk:
        lk.loglik(theta, srw.SRW_FP32, out=out)
        torch.cuda.synchronize()
        assert np.all(np.isposinf(out.cpu().numpy()))


# FP32 products: the tile that a batch gets depends on its size, the value of a
# point does not.
@pytest.mark.parametrize("n_t,n_rec,p", [(100, 64, 9800), (64, 129, 4900), (260, 200, 4900), (33, 1111, 1200),
                                         (300, 2050, 640)])
def test_fp32_value_independent_of_the_batch(srw, n_t, n_rec, p):
    wl = line(n_t, n_rec)
    _, counts = oracle_of(wl)
    theta = workloads.theta_box(p, 11)
    with srw.Likelihood(wl, counts) as lk:
        want, spec = lk.loglik(theta, srw.SRW_FP32), lk.spectrum_batch(theta, srw.SRW_FP32)
        for k in (2, 31, 33, 65, 300):
            np.testing.assert_array_equal(lk.loglik(theta[:k], srw.SRW_FP32), want[:k])
            np.testing.assert_array_equal(lk.spectrum_batch(theta[:k], srw.SRW_FP32), spec[:k])


# No room for the FP32 batch's copy of R: the handle is made all the same, and the
# batch makes the copy when it is called.
def test_create_without_room_for_the_fp32_copy(srw):
    wl = line(64, 130)
    m, counts = oracle_of(wl)
    theta = workloads.fit_region_points(4, seed=7)
    want = m.neg2lnl_batch(theta.astype(np.float64))
    made = 0
    for skip in range(100):
        srw.srw_fault_inject("alloc", skip)
        try:
            lk = srw.Likelihood(wl)
        except srw.SrwError as e:
            assert e.status == 2  # SRW_ENOMEM
            continue
        fired = srw.srw_fault_pending() == 0
        srw.srw_fault_inject("none")
        srw.srw_set_data(lk.handle, counts, wl["bkg"])
        assert np.max(np.abs(lk.loglik(theta, srw.SRW_FP32) - want)) <= 1e-4
        lk.close()
        if not fired:  # past the last allocation
            break
        made += 1
    assert made == 2  # either of the two copies


# Page-locked host memory serves host-pointer calls: handles that make none hold none.
def test_handles_pin_no_host_memory_before_a_host_call(srw):
    def shared_kb():
        with open("/proc/self/status") as f:
            return sum(int(x.split()[1]) for x in f if x.startswith("RssShmem"))

    wl = line(64, 130)
    _, counts = oracle_of(wl)
    theta = torch.zeros((1, 5), device="cuda")
    first = srw.Likelihood(wl, counts)  # whatever the process maps once
    first.loglik(theta, out=torch.zeros(1, dtype=torch.float64, device="cuda"))
    before = shared_kb()
    rest = [srw.Likelihood(wl, counts) for _ in range(32)]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    for lk in rest:
        lk.loglik(theta, out=out)
    assert shared_kb() - before < 32 * 64
    want = first.loglik(np.zeros((1, 5), np.float32))
    for lk in rest:
        np.testing.assert_array_equal(lk.loglik(np.zeros((1, 5), np.float32)), want)
        lk.close()
    first.close()


# Surrogate: a full chunk and a small batch cut the bins into different units.
@pytest.mark.parametrize("n_rec", [100, 257, 600, 1000, 1300, 2048, 4000])
def test_surrogate_value_independent_of_the_batch(srw, n_rec):
    from workloads.mlp import BOX_CENTRE, BOX_HALF, init_weights
    wl = line(64, n_rec)
    _, counts = oracle_of(wl)
    params = init_weights(n_rec, seed=5)
    # neighbouring bins of one size between exp(-25) and exp(18): the sums of 16 bins round where they are added up
    bias = np.repeat(np.random.default_rng(n_rec).uniform(-25.0, 18.0, n_rec // 16 + 1), 16)[:n_rec].astype(np.float32)
    params[-1] = (0.1 * params[-1][0], bias)
    theta = workloads.theta_box(100000, 43)
    with srw.Likelihood(wl, counts) as lk, srw.Surrogate(lk, params, BOX_CENTRE, BOX_HALF) as s:
        v = s.loglik(theta)
        assert np.all(np.isfinite(v))
        for p in (1, 257, 3000, 20000, 40000):
            np.testing.assert_array_equal(s.loglik(theta[:p]), v[:p])


# Rank 8: an empty bin with a subnormal expectation shares the warps' rounds with
# ordinary bins; the value of a point does not depend on the path of its batch.
@pytest.mark.parametrize("n_rec", [65, 257])
def test_rank8_empty_bins_beside_ordinary_ones(srw, n_rec):
    wl = line(50, n_rec)
    r, bkg = wl["R"].copy(), wl["bkg"].copy()
    _, counts = oracle_of(wl)
    for j in range(1, n_rec, 9):
        r[j], bkg[:, j], counts[j] = 0.0, 1e-35, 0.0
    wl.update(R=r, bkg=bkg)
    theta = workloads.fit_region_points(19456, seed=5)
    with srw.Likelihood(wl, counts) as lk:
        v, g = lk.loglik_linear(theta, grad=True)
        assert np.all(np.isfinite(v)) and np.all(np.isfinite(g))
        np.testing.assert_array_equal(lk.loglik_linear(theta), v)
        for p in (1, 16, 2433, 9728):
            v1, g1 = lk.loglik_linear(theta[:p], grad=True)
            np.testing.assert_array_equal(v1, v[:p])
            np.testing.assert_array_equal(g1, g[:p])


# Two million reconstructed bins: more rows than a grid's y dimension holds in tiles of 32.
def test_fp32_batch_with_very_many_bins(srw):
    from scipy.special import gammaln, xlogy
    n_rec, n_t = 2100001, 2
    rng = np.random.default_rng(1)
    r = rng.uniform(0.5, 1.5, (n_rec, n_t)).astype(np.float32) / np.float32(n_rec)
    wl = line(n_t, 8)
    wl.update(R=r[:8], e_true_sm=np.full(n_t, 1.0e6))
    m = O.OracleModel.from_workload(wl, e_true_sm=wl["e_true_sm"])  # spectra only: the fold is one product here
    bkg = rng.uniform(0.5, 1.0, (1, n_rec))
    ref = r.astype(np.float64) @ m.weighted_true(np.zeros(5)) + bkg[0]
    counts = rng.poisson(ref).astype(np.float64)
    wl.update(R=r, rec_edges=np.linspace(0.0, 1.3, n_rec + 1), bkg=bkg)
    theta = workloads.fit_region_points(2, seed=3)
    with srw.Likelihood(wl, counts, e_true_sm=wl["e_true_sm"]) as lk:
        got = lk.loglik(theta, srw.SRW_FP32)
    for t, v in zip(theta, got):
        mu = r.astype(np.float64) @ m.weighted_true(t.astype(np.float64)) + bkg[0]
        want = 2.0 * np.sum(mu - xlogy(counts, mu) + gammaln(counts + 1.0))
        # FP32 products of R with the deviation from the reference: 2^-23 of each
        assert abs(v - want) <= 2.0 * np.sum(np.abs(1.0 - counts / mu) * np.abs(mu - ref)) * 2.0**-23


# The first pass at a batch size fills its input buffer's padding and runs at once:
# its values are those of the second pass (a fill of 256 MB is still on its way
# when the next launch is made).
def test_surrogate_first_pass_of_a_large_batch(srw):
    from workloads.mlp import BOX_CENTRE, BOX_HALF, init_weights
    wl = line(64, 100)
    _, counts = oracle_of(wl)
    theta = torch.from_numpy(workloads.theta_box(1 << 20, 43)).cuda()
    with srw.Likelihood(wl, counts) as lk:
        for _ in range(3):
            with srw.Surrogate(lk, init_weights(100, seed=5), BOX_CENTRE, BOX_HALF) as s:
                first, second = (torch.zeros(1 << 20, dtype=torch.float64, device="cuda") for _ in range(2))
                s.loglik(theta, out=first)
                s.loglik(theta, out=second)
                torch.cuda.synchronize()
                assert torch.equal(first, second)


# A device wait that runs out in a surrogate pass: no value, never an earlier call's.
# The sizes give each form of the partial sums: of short units, of runs, of quarters.
@pytest.mark.parametrize("skip", [0, 1, 2, 3])
@pytest.mark.parametrize("n_rec,p", [(300, 300), (300, 3000), (2048, 20000), (100, 100000)])
def test_surrogate_timeout_gives_no_value(srw, n_rec, p, skip):
    from workloads.mlp import BOX_CENTRE, BOX_HALF, init_weights
    wl = line(64, n_rec)
    _, counts = oracle_of(wl)
    with srw.Likelihood(wl, counts) as lk, srw.Surrogate(lk, init_weights(n_rec, seed=5), BOX_CENTRE, BOX_HALF) as s:
        theta = workloads.theta_box(p, 43)
        other = workloads.theta_box(p, 44)
        want = s.loglik(theta)
        s.loglik(other)  # the buffers hold another call's partial sums
        dev, out = torch.from_numpy(theta).cuda(), torch.zeros(p, dtype=torch.float64, device="cuda")
        srw.srw_fault_inject("timeout", skip)  # one of the pass's four kernels
        s.loglik(dev, out=out)
        torch.cuda.synchronize()
        assert srw.srw_fault_pending() == 0
        got = out.cpu().numpy()
        bad = np.isnan(got)
        assert bad.any()
        np.testing.assert_array_equal(got[~bad], want[~bad])
        with pytest.raises(srw.SrwError) as ei:  # the next host call reads and clears the status
            s.loglik(other)
        assert ei.value.status == 6  # SRW_ETIMEOUT
        np.testing.assert_array_equal(s.loglik(theta), want)
