"""CUDA path vs the FP64 oracle, element by element, through the C ABI.

Tolerances (from the workload definition): FP64 mode 1e-9 relative on chi^2,
mu and spectra and 1e-9 normwise on the gradient; mixed modes 1e-6 relative on
P, mu, spectra and chi^2 (gradient reported with a loose 1e-4 sanity bound).
chi^2 is held to the plain relative tolerance and, in addition, to the same
tolerance scaled by max(chi2, sum_i |g_i| mu_i) -- the largest chi^2 change a
relative change of every mu_i can cause.  Two mixed-precision cases keep only
the scaled bound, each with its measured reason at the test: bins of 3-16
nodes, and one bin whose chi^2 is 338x below that scale.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1804_07682_gb300 import _native as N
from paper_1804_07682_gb300 import workloads as wl
from refs import Case, check_chi2, fit_sigma, log_err, normrel, rel

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

TOL = {"fp64": 1e-9, "f64phase": 1e-6, "ff": 1e-6}
GTOL = {"fp64": 1e-9, "f64phase": 1e-4, "ff": 1e-4}


@pytest.fixture(scope="module")
def api():
    from paper_1804_07682_gb300 import api as _api
    return _api


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def make_plan(api, case, prec, mapping=None, with_plain=False, per_point_data=False):
    w = case.w
    return api.Plan(w.edges, w.L, nodes_per_bin=w.nodes_per_bin, npts=w.npts, node_counts=w.node_counts,
                    norm=case.N, e_scale=w.e_scale, prec=prec, kind=w.kind,
                    max_datasets=w.npts if per_point_data else 0, with_plain=with_plain, mapping=mapping)


# ------------------------------------------------------------ Gauss-Legendre
@pytest.mark.parametrize("n", [1, 2, 3, 7, 50, 262, 524, 4096, 16384, 65536])
def test_gl_nodes(api, n):
    x, w = api.gl_nodes(n)
    xr, wr = oracle.gl(n)
    x = x.cpu().numpy()
    assert np.abs(x - xr).max() < 2e-15
    # a one-ulp difference in a node moves its weight by ~4|x|/(1-x^2) ulp;
    # the weight needs P_n' from an n-step three-term recurrence, which the
    # two sides round differently (up to ~n ulp: at n = 65536 the oracle and
    # a float64 replay of the kernel's recurrence are within 8e-12 of 40-digit
    # weights at sampled nodes, and the two sides measured 4.8e-12 apart)
    eps = np.spacing(1.0)
    tol = 1e-12 + n * eps + 4 * eps * np.abs(xr) / ((1 - xr) * (1 + xr))
    assert np.all(np.abs(w.cpu().numpy() / wr - 1) <= tol)


# ------------------------------------------------------------------ OscProb
@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
@pytest.mark.parametrize("rng_case", ["reactor", "long_baseline", "largest_phases"])
def test_oscprob(api, prec, rng_case):
    rng = np.random.default_rng(11)
    if rng_case == "reactor":
        E = rng.uniform(0.5, 15.0, 100003)
        L = [0.5, 52.5, 60.0, 17.3]
    elif rng_case == "largest_phases":
        # reactor energies across the Earth: Delta_31 up to 9.4e3 rad, near
        # the 12,868 rad below which the double-float phase's reduction is exact
        E = rng.uniform(1.8, 15.0, 100003)
        L = [3000.0, 5200.0]
    else:
        E = rng.uniform(500.0, 5000.0, 4099)
        L = [810.0]
    theta = (0.307, 0.0218, 7.53e-5, 2.44e-3 * 1.05)
    P = api.oscprob(dev(E), L, theta, prec).double().cpu().numpy()
    for r, Lr in enumerate(L):
        ref = oracle.pee(E, Lr, theta)
        assert rel(P[r], ref) < (1e-10 if prec == "fp64" else TOL[prec]), (prec, Lr)


@pytest.mark.parametrize("prec", ["fp64", "ff"])
def test_oscprob_reads_and_writes_pinned_host_memory(api, prec):
    # energies and probabilities in pinned host memory, used in place by the kernels
    rng = np.random.default_rng(12)
    E = rng.uniform(0.5, 15.0, 200003)
    Eh = torch.as_tensor(E).pin_memory()
    Ph = api.oscprob(Eh, [52.5, 1.0], wl.TRUTH, prec)
    Pd = api.oscprob(dev(E), [52.5, 1.0], wl.TRUTH, prec)
    torch.cuda.synchronize()
    assert not Ph.is_cuda and Ph.is_pinned()
    assert torch.equal(Ph, Pd.cpu())
    th = (0.307, 0.0218, 0.545, 1.2 * np.pi, 7.53e-5, 2.44e-3)
    Gh = api.oscprob_general(Eh, [810.0], th, "mu", "e", prec=prec)
    Gd = api.oscprob_general(dev(E), [810.0], th, "mu", "e", prec=prec)
    torch.cuda.synchronize()
    assert torch.equal(Gh, Gd.cpu())
    with pytest.raises(ValueError):
        api.oscprob(torch.as_tensor(E), [52.5], wl.TRUTH, prec)  # pageable host memory is refused


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("n,chunk", [(200003, 0), (200003, 65536), (200003, 7), (1000, 4096), (1, 0), (70001, 70000)])
def test_oscprob_staged_chunks(api, prec, n, chunk):
    # host to host through device staging in chunks (ragged last chunk, chunk
    # larger than n, more chunks than stages): identical to the device result
    rng = np.random.default_rng(n + chunk)
    E = rng.uniform(0.5, 15.0, n)
    if chunk == 7:
        E = E[:5000]
    Eh = torch.as_tensor(E).pin_memory()
    Ph = api.oscprob_staged(Eh, [52.5, 1.0, 0.0], wl.TRUTH, prec, chunk=chunk)
    Pd = api.oscprob(dev(E), [52.5, 1.0, 0.0], wl.TRUTH, prec)
    torch.cuda.current_stream().synchronize()
    assert Ph.is_pinned() and torch.equal(Ph, Pd.cpu())


def test_oscprob_staged_refuses_unpinned(api):
    E = torch.linspace(1.0, 10.0, 100, dtype=torch.float64)
    with pytest.raises(ValueError):
        api.oscprob_staged(E, [52.5], wl.TRUTH)
    with pytest.raises(ValueError):
        api.oscprob_staged(E.cuda(), [52.5], wl.TRUTH)
    # the C ABI itself refuses device memory for the host arguments
    Ed = E.cuda()
    Pd = torch.empty(1, 100, dtype=torch.float64, device="cuda")
    p = N.GnaOsc(*wl.TRUTH)
    L = np.array([52.5])
    code = N.lib().gna_oscprob_ee_staged(ctypes.c_void_p(Ed.data_ptr()), 100,
                                         L.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 1, ctypes.byref(p),
                                         0, ctypes.c_void_p(Pd.data_ptr()), 0, None)
    assert code == 1  # GNA_EINVAL
    # and pointers that are not aligned to their element type (refused on the
    # host, before any launch)
    Eh = torch.linspace(1.0, 10.0, 101, dtype=torch.float64).pin_memory()
    Ph = torch.empty(1, 101, dtype=torch.float64).pin_memory()
    Lp = L.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    code = N.lib().gna_oscprob_ee_staged(ctypes.c_void_p(Eh.data_ptr() + 4), 100, Lp, 1, ctypes.byref(p), 0,
                                         ctypes.c_void_p(Ph.data_ptr()), 0, None)
    assert code == 1
    Ed = torch.linspace(1.0, 10.0, 101, dtype=torch.float64, device="cuda")
    code = N.lib().gna_oscprob_ee(ctypes.c_void_p(Ed.data_ptr() + 4), 100, Lp, 1, ctypes.byref(p), 0,
                                  ctypes.c_void_p(Pd.data_ptr()), None)
    assert code == 1


def test_oscprob_edge_cases(api):
    E = dev([3.0])
    P = api.oscprob(E, [0.0, 52.5], wl.TRUTH, "ff").cpu().numpy()
    assert P[0, 0] == 1.0
    assert abs(P[1, 0] - oracle.pee([3.0], 52.5, wl.TRUTH)[0]) < 1e-6
    assert api.oscprob(dev(np.zeros(0)), [1.0], wl.TRUTH, "fp64").numel() == 0


# ------------------------------------------------- OscProb, any channel
THETA_FULL = (0.307, 0.0218, 0.545, 1.2 * np.pi, 7.53e-5, 2.44e-3)
FL = {"e": 0, "mu": 1, "tau": 2}


def oracle_prob(a, b, E, L, anti, th=THETA_FULL):
    s12, s13, s23, d, dm21, dm32 = th
    return np.array([oracle.prob(FL[a], FL[b], s12, s13, s23, d, dm21, dm32, L, e, anti) for e in E])


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
@pytest.mark.parametrize("anti", [False, True])
@pytest.mark.parametrize("a,b", [("e", "e"), ("mu", "mu"), ("mu", "e"), ("e", "tau"), ("tau", "mu")])
def test_oscprob_general(api, prec, anti, a, b):
    # long-baseline energies (0.5-5 GeV) at 810 and 295 km, the Im (CP) term on
    rng = np.random.default_rng(5)
    E = rng.uniform(500.0, 5000.0, 1537)
    L = [810.0, 295.0]
    P = api.oscprob_general(dev(E), L, THETA_FULL, a, b, anti=anti, prec=prec).double().cpu().numpy()
    for r, Lr in enumerate(L):
        ref = oracle_prob(a, b, E, Lr, anti)
        err = np.abs(P[r] - ref).max()
        assert err < (1e-12 if prec == "fp64" else 3e-7), (prec, a, b, anti, Lr, err)


def test_oscprob_general_identities(api):
    rng = np.random.default_rng(6)
    E = dev(rng.uniform(200.0, 8000.0, 4099))
    L = [810.0, 52.5, 0.0]
    P = {(a, b, anti): api.oscprob_general(E, L, THETA_FULL, a, b, anti=anti).cpu().numpy()
         for a in FL for b in FL for anti in (False, True)}
    for anti in (False, True):
        for a in FL:  # unitarity: rows and columns sum to one
            assert np.abs(sum(P[(a, b, anti)] for b in FL) - 1.0).max() < 1e-12
            assert np.abs(sum(P[(b, a, anti)] for b in FL) - 1.0).max() < 1e-12
    for a in FL:  # CPT: P(a -> b, antineutrino) = P(b -> a, neutrino)
        for b in FL:
            assert np.abs(P[(a, b, True)] - P[(b, a, False)]).max() < 1e-13
            assert np.all(P[(a, b, False)][2] == (1.0 if a == b else 0.0))  # L = 0
    # nue_bar survival from the general kernel equals the dedicated one
    th4 = (THETA_FULL[0], THETA_FULL[1], THETA_FULL[4], THETA_FULL[5])
    Pee = api.oscprob(E, L, th4, "fp64").cpu().numpy()
    assert np.abs(P[("e", "e", True)] - Pee).max() < 1e-13
    from paper_1804_07682_gb300 import _native as N
    with pytest.raises(N.GnaError):
        api.oscprob_general(E, L, THETA_FULL, 3, 0)


# ------------------------------------------------------- chain, small cases
def small_cases():
    return {
        "reactor_200x50": lambda: wl.reactor_200x50(),
        "reactor8_40x3000": lambda: wl.shrink(wl.reactor8_1000x16384(), nbins=40, nodes=3000),
        "nuisance_64x1000": lambda: wl.shrink(wl.nuisance_1000x4096(), nbins=64, nodes=1000),
        "scan_16pts_60bins": lambda: wl.shrink(wl.scan_64x64_500bins(4, 4), nbins=60),
        "fits_8x100x20": lambda: wl.shrink(wl.fits_16384x1000(8), nbins=100, nodes=20),
    }


_case_cache = {}


def get_case(name):
    if name not in _case_cache:
        w = small_cases()[name]()
        tn = None if name != "scan_16pts_60bins" else 64
        _case_cache[name] = Case(w, truth_nodes=tn)
    return _case_cache[name]


def check_chain(api, case, prec, mapping=None, spectra=True, plain_chi2=True):
    w = case.w
    per_point = case.data.ndim == 2
    plan = make_plan(api, case, prec, mapping, per_point_data=per_point)
    eta = None if w.eta is None else dev(w.eta)
    out = plan.eval(plan.params_tensor(w.theta), dev(case.data), eta, w.sigma_eta, grad=True,
                    grad_eta=eta is not None, mu=True, spectra=spectra)
    torch.cuda.synchronize()
    plan.status()
    tol, gtol = TOL[prec], GTOL[prec]
    for p in range(w.npts):
        ref = case.oracle_point(p)
        check_chi2(out["chi2"][p].item(), ref, case.data_of(p), w.kind, tol, tag="chain %s %s %s p%d" % (
            w.name, prec, mapping, p), plain=plain_chi2)
        assert rel(out["mu"][p].cpu().numpy(), ref["mu"]) < tol
        if spectra:
            assert rel(out["spectra"][p].cpu().numpy(), ref["mu_rb"]) < tol
        assert normrel(out["grad"][p].cpu().numpy(), ref["grad"][:4]) < gtol
        if eta is not None:
            assert normrel(out["grad_eta"][p].cpu().numpy(), ref["grad"][4:]) < gtol
    plan.close()


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
@pytest.mark.parametrize("name", list(small_cases()))
def test_chain_small(api, name, prec):
    check_chain(api, get_case(name), prec)


@pytest.mark.parametrize("mapping", ["split", "bins", "slices"])
@pytest.mark.parametrize("name", ["reactor_200x50", "reactor8_40x3000", "fits_8x100x20"])
def test_chain_all_mappings(api, name, mapping):
    check_chain(api, get_case(name), "ff", mapping)


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("tuning", ["slice=16", "slice=7", "slice=100 block=64", "slice=3000 block=128", "slice=999"])
def test_slice_shapes(api, prec, tuning):
    # slices of 7 ... 3000 nodes of 3000-node bins (ragged last slice), spectra on
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, prec, "slices")
    plan.tuning = tuning
    out = plan.eval(plan.params_tensor(w.theta), dev(case.data), grad=True, mu=True, spectra=True)
    ref = case.oracle_point(0)
    tol = TOL[prec]
    check_chi2(out["chi2"][0].item(), ref, case.data, w.kind, tol, tag="slice_shapes %s %s" % (prec, tuning))
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < tol
    assert rel(out["spectra"][0].cpu().numpy(), ref["mu_rb"]) < tol
    assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:4]) < GTOL[prec]
    plan.close()


@pytest.mark.parametrize("tuning", ["block=64 nodes=4", "block=128 nodes=7", "block=256 nodes=64", "block=96 nodes=5",
                                    "block=256 nodes=1024", "block=32 nodes=4 grid=1"])
def test_chain_launch_shapes(api, tuning):
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, "ff", "split")
    plan.tuning = tuning
    out = plan.eval(plan.params_tensor(w.theta), dev(case.data), grad=True, mu=True)
    ref = case.oracle_point(0)
    assert rel(out["chi2"][0].item(), ref["chi2"]) < 1e-6
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < 1e-6


@pytest.mark.parametrize("mapping,tuning", [("split", "block=64 nodes=4"), ("slices", "block=64 slice=20")])
def test_repeated_evaluations_are_bit_identical(api, mapping, tuning):
    # segment and slice values are summed in slot order and the point sums in
    # bin order, whatever order the warps finish in
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, "ff", mapping)
    plan.tuning = tuning
    p = plan.params_tensor(w.theta)
    d = dev(case.data)
    outs = [{k: v.clone() for k, v in plan.eval(p, d, grad=True, mu=True, spectra=True).items()} for _ in range(6)]
    for o in outs[1:]:
        for k in o:
            assert torch.equal(o[k], outs[0][k]), k
    plan.close()


def test_chain_degenerate_shapes(api):
    # one bin, one node per bin, one baseline; and zero-count bins in the data
    w = wl.Workload("one", np.array([2.0, 2.5]), 1, np.array([52.5]), np.array([wl.TRUTH]), wl.POISSON)
    case = Case(w)
    case.data = np.array([0.0])
    for prec in ("fp64", "ff"):
        check_chain(api, case, prec)
    w2 = wl.shrink(wl.reactor8_1000x16384(), nbins=33, nodes=1)
    case2 = Case(w2)
    for prec in ("fp64", "ff"):
        check_chain(api, case2, prec)


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
def test_chain_boundary_parameters(api, prec):
    # points on the edges of the physical domain: theta13 = 0 (two-flavour
    # limit), theta12 = 0 and 90 degrees, dm2_21 = 0, theta13 = 90 degrees
    # (P = 1), and a vanishing dm2_32; reactor bins, eight baselines
    t = wl.TRUTH
    theta = np.array([[t[0], 0.0, t[2], t[3]], [0.0, t[1], t[2], t[3]], [1.0, t[1], t[2], t[3]],
                      [t[0], t[1], 0.0, t[3]], [t[0], 1.0, t[2], t[3]], [t[0], t[1], t[2], 1e-9]])
    w = wl.Workload("boundary", np.linspace(1.8, 12.0, 41), 24, wl.reactor8_1000x16384().L, theta, wl.POISSON)
    check_chain(api, Case(w), prec)


@pytest.mark.parametrize("kind", [wl.PEARSON, wl.POISSON])
@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
def test_chain_sparse_counts(api, prec, kind):
    # 300 events over the 200 reactor bins (8 baselines): Poisson data with
    # many empty bins (the d = 0 terms of both chi^2 kinds)
    w = wl.Workload("sparse", np.linspace(1.8, 12.0, 201), 50, wl.reactor8_1000x16384().L,
                    np.array([wl.TRUTH]) * np.array([[1.02, 0.97, 1.01, 0.99]]), kind)
    case = Case(w)
    scale = 300.0 / case.mu_truth.sum()
    case.N *= scale
    case.mu_truth = case.mu_truth * scale
    case.data = wl.poisson_data(case.mu_truth, 77)
    assert np.sum(case.data == 0) > 20
    check_chain(api, case, prec)


@pytest.mark.parametrize("mapping", ["split", "bins", "slices"])
@pytest.mark.parametrize("nbins,n,npts", [(1, 8, 40), (3, 5, 50), (2, 16, 3), (7, 3, 33), (2, 40, 3)])
def test_grids_shorter_than_a_warp(api, nbins, n, npts, mapping):
    # the whole grid (bins x nodes) has fewer nodes than a warp has lanes, so a
    # lane's next node lies several bins, or several points, further on
    rng = np.random.default_rng(nbins * 100 + n)
    theta = np.tile(np.array(wl.TRUTH), (npts, 1)) * rng.uniform(0.9, 1.1, size=(npts, 4))
    w = wl.Workload("tiny", np.linspace(2.0, 8.0, nbins + 1), n, np.array([52.5, 53.0]), theta, wl.POISSON)
    case = Case(w)
    # bins of 3-16 nodes: in the mixed precisions a node's P carries ~1e-7 of
    # FP32 rounding that so few nodes cannot average, and chi^2 here is 36-54x
    # below its error scale sum_i |g_i| mu_i (measured up to 6.8e-6 relative):
    # the scaled bound only; GNA_FP64 keeps the plain relative 1e-9
    for prec in (("f64phase", "ff") if mapping == "slices" else ("fp64", "ff")):
        check_chain(api, case, prec, mapping, plain_chi2=(prec == "fp64"))


@pytest.mark.parametrize("nL", [3, 5, 12, 16])
@pytest.mark.parametrize("prec,mapping", [("fp64", None), ("ff", "split"), ("ff", "bins"), ("ff", "slices")])
def test_baseline_counts_between_instantiations(api, nL, prec, mapping):
    # kernels exist for 1, 2, 4, 8 and 16 baselines; other counts run the next
    # one up with zero-weight padding, and their per-baseline spectra must
    # still be those of the real baselines only
    rng = np.random.default_rng(nL)
    L = np.sort(rng.uniform(0.5, 60.0, nL))
    theta = np.array([wl.TRUTH]) * rng.uniform(0.97, 1.03, size=(1, 4))
    w = wl.Workload("baselines_%d" % nL, np.linspace(1.8, 9.0, 41), 24, L, theta, wl.POISSON)
    check_chain(api, Case(w), prec, mapping)


@pytest.mark.parametrize("prec,mapping", [("fp64", None), ("ff", "split"), ("ff", "bins"), ("ff", "slices")])
def test_many_bins(api, prec, mapping):
    # 40001 bins (1251 groups of 32, the last holding one bin) of 3 nodes
    theta = np.array([wl.TRUTH])
    w = wl.Workload("many_bins", np.linspace(1.8, 12.0, 40002), 3, np.array([52.5, 1.5]), theta, wl.PEARSON)
    check_chain(api, Case(w), prec, mapping)


@pytest.mark.parametrize("prec,mapping", [("fp64", None), ("ff", "split"), ("ff", "slices"), ("f64phase", "slices")])
def test_one_bin_of_many_nodes(api, prec, mapping):
    # one bin (one lane of one group busy) of 16384 nodes, eight baselines:
    # the slice mapping cuts it into its largest number of slices.  Its chi^2
    # (3.5) is 338x below sum |g| mu, so the mixed precisions' 4e-9 relative
    # error of mu shows as 1.4e-6 on chi^2 (measured): the scaled bound there
    w = wl.shrink(wl.reactor8_1000x16384(), nbins=1)
    check_chain(api, Case(w), prec, mapping, plain_chi2=(prec == "fp64"))


_largest = {}


@pytest.mark.parametrize("prec,mapping", [("fp64", None), ("ff", "slices"), ("ff", "bins")])
def test_one_bin_of_the_largest_order(api, prec, mapping):
    # the same bin at the largest Gauss-Legendre order a plan accepts (65536
    # nodes): grid build at that order and the longest node loops; chi^2 as
    # in the 16384-node case (scaled bound in the mixed modes)
    if "case" not in _largest:
        w = wl.shrink(wl.reactor8_1000x16384(), nbins=1)
        _largest["case"] = Case(wl.Workload("one_bin_65536", w.edges, 65536, w.L, w.theta, w.kind))
    check_chain(api, _largest["case"], prec, mapping, plain_chi2=(prec == "fp64"))


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
def test_points_sharing_grids(api, prec):
    # points with equal node counts share one energy grid on the device; the
    # counts are interleaved so that a shared grid serves points far apart in
    # the point order, and the largest count is held by a single point
    rng = np.random.default_rng(5)
    counts = np.array([7, 12, 7, 30, 12, 7, 5, 30, 12, 41])
    theta = np.tile(np.array(wl.TRUTH), (counts.size, 1)) * rng.uniform(0.95, 1.05, size=(counts.size, 4))
    w = wl.Workload("shared_grids", np.linspace(1.8, 8.0, 71), 0, np.array([52.5, 53.1]), theta, wl.POISSON,
                    node_counts=counts)
    check_chain(api, Case(w), prec)


@pytest.mark.parametrize("name", ["reactor8_40x3000", "scan_16pts_60bins", "fits_8x100x20", "nuisance_64x1000",
                                  "reactor_200x50"])
def test_plain_chain_matches_oracle(api, name):
    # the plain FP64 one-kernel-per-transformation chain: eight baselines,
    # uneven per-point grids (16 points, points sharing grids), one data row
    # per point, nuisances; every point against the oracle at 1e-9
    case = get_case(name)
    w = case.w
    per_point = case.data.ndim == 2
    plan = make_plan(api, case, "ff", with_plain=True, per_point_data=per_point)
    eta = None if w.eta is None else dev(w.eta)
    out = plan.eval(plan.params_tensor(w.theta), dev(case.data), eta, w.sigma_eta, grad=True,
                    grad_eta=eta is not None, mu=True, spectra=True, plain=True)
    torch.cuda.synchronize()
    plan.status()
    assert plan.launches == 1 + 6  # prepare, then one chunk of six kernels
    for p in range(w.npts):
        ref = case.oracle_point(p)
        check_chi2(out["chi2"][p].item(), ref, case.data_of(p), w.kind, 1e-9, tag="plain %s p%d" % (name, p))
        assert rel(out["mu"][p].cpu().numpy(), ref["mu"]) < 1e-9
        assert rel(out["spectra"][p].cpu().numpy(), ref["mu_rb"]) < 1e-9
        assert normrel(out["grad"][p].cpu().numpy(), ref["grad"][:4]) < 1e-9
        if eta is not None:
            assert normrel(out["grad_eta"][p].cpu().numpy(), ref["grad"][4:]) < 1e-9
    plan.close()


def test_sampled_kernel_profiling(api):
    case = get_case("reactor_200x50")
    w = case.w
    plan = make_plan(api, case, "ff")
    p, d = plan.params_tensor(w.theta), dev(case.data)
    plan.profile(3)  # evaluations 0, 3, 6 and 9 of ten are timed
    for _ in range(10):
        plan.eval(p, d, grad=True)
    ms, n = plan.profile_read()
    assert n == 4 and ms > 0.0
    plan.profile(0)
    plan.eval(p, d, grad=True)
    assert plan.profile_read() == (0.0, 0)
    from paper_1804_07682_gb300 import _native as N
    with pytest.raises(N.GnaError):
        plan.profile(-1)
    plan.close()


def test_graph_replay_and_host_buffers(api):
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, "ff")
    p = plan.params_tensor(w.theta)
    d = dev(case.data)
    a = plan.eval(p, d, grad=True)
    a = {k: v.clone() for k, v in a.items()}
    plan.set_graph(True)
    outs = {"chi2": torch.empty(1, dtype=torch.float64, device="cuda"),
            "grad": torch.empty(1, 4, dtype=torch.float64, device="cuda")}
    for _ in range(3):
        plan.eval(p, d, grad=True, out=outs)
    torch.cuda.synchronize()
    assert torch.equal(outs["chi2"], a["chi2"]) and torch.equal(outs["grad"], a["grad"])
    assert plan.launches >= 2
    c, g = plan.eval_host(w.theta, case.data, grad=True)
    assert c[0] == a["chi2"][0].item() and np.array_equal(g, a["grad"].cpu().numpy())


@pytest.mark.parametrize("graph", [False, True])
def test_host_evaluations_pipelined(api, graph):
    # two outstanding host evaluations with different inputs, taken in order,
    # give the same results as one synchronous call each; a third is refused
    from paper_1804_07682_gb300 import _native as N
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, "ff")
    plan.set_graph(graph)
    th0 = np.asarray(w.theta, dtype=np.float64).reshape(1, 4)
    th1 = th0 * np.array([[1.01, 0.99, 1.02, 0.995]])
    spec = np.empty((1, w.nL, w.nbins))
    ref0 = plan.eval_host(th0, case.data, grad=True, spectra_out=spec.copy())  # same kernel as t0 (spectra on)
    ref1 = plan.eval_host(th1, case.data, grad=True)
    for _ in range(3):
        t0 = plan.eval_host_async(th0, case.data, grad=True, spectra=True)
        t1 = plan.eval_host_async(th1, case.data, grad=True)
        with pytest.raises(N.GnaError):
            plan.eval_host_async(th0, case.data)
        c0, g0 = plan.eval_host_wait(t0, spectra_out=spec)
        with pytest.raises(N.GnaError):
            plan.eval_host_wait(t0)
        c1, g1 = plan.eval_host_wait(t1)
        assert c0[0] == ref0[0][0] and np.array_equal(g0, ref0[1])
        assert c1[0] == ref1[0][0] and np.array_equal(g1, ref1[1])
    ref = case.oracle_point(0)
    assert rel(spec[0], ref["mu_rb"]) < 1e-6
    plan.close()


@pytest.mark.parametrize("mapping", ["split", "bins", "slices"])
def test_cached_epilogue_matches_full_evaluation(api, mapping):
    # new nuisances and new data on the kept node sums give exactly what a
    # full evaluation with them gives (same sums, same epilogue)
    from paper_1804_07682_gb300 import _native as N
    case = get_case("nuisance_64x1000")
    w = case.w
    plan = make_plan(api, case, "ff", mapping)
    p = plan.params_tensor(w.theta)
    d = dev(case.data)
    with pytest.raises(N.GnaError):
        plan.eval_cached(d, dev(w.eta), w.sigma_eta)  # nothing kept yet
    kw = dict(grad=True, grad_eta=True, mu=True, spectra=True)
    plan.eval(p, d, dev(w.eta), w.sigma_eta, **kw)
    rng = np.random.default_rng(8)
    eta2 = dev(rng.normal(0.0, 0.02, w.nbins))
    d2 = dev(rng.poisson(case.data).astype(np.float64))
    for eta_c, d_c in ((eta2, d), (eta2, d2), (dev(w.eta), d2)):
        c = {k: v.clone() for k, v in plan.eval_cached(d_c, eta_c, w.sigma_eta, **kw).items()}
        f = plan.eval(p, d_c, eta_c, w.sigma_eta, **kw)
        for k in c:
            assert torch.equal(c[k], f[k]), (mapping, k)
    # against the oracle too, for the last pair
    ref = oracle.chain(w.edges, w.nodes_per_bin, w.L, w.theta[0], case.N, d2.cpu().numpy(), w.kind, eta=w.eta,
                       sigma=w.sigma_eta)
    check_chi2(c["chi2"][0].item(), ref, d2.cpu().numpy(), w.kind, 1e-6, tag="cached " + mapping)
    assert rel(c["mu"][0].cpu().numpy(), ref["mu"]) < 1e-6
    # kept without a gradient: a gradient is refused, chi^2 alone is fine
    plan.eval(p, d, grad=False)
    with pytest.raises(N.GnaError):
        plan.eval_cached(d, grad=True)
    plan.eval_cached(d, grad=False)
    plan.close()


def test_autotune_keeps_parity(api):
    case = get_case("reactor8_40x3000")
    w = case.w
    plan = make_plan(api, case, "ff")
    p = plan.params_tensor(w.theta)
    d = dev(case.data)
    text = plan.autotune(p, d, reps=2)
    assert "block=" in text
    out = plan.eval(p, d, grad=True)
    ref = case.oracle_point(0)
    assert rel(out["chi2"][0].item(), ref["chi2"]) < 1e-6


@pytest.mark.parametrize("prec", ["fp64", "ff"])
def test_mapping_is_a_tuning_choice_on_small_grids(api, prec):
    # a small uniform grid keeps both layouts: the two mappings give the same
    # answer from one plan, and the autotuner (timing graph replays) may pick either
    case = get_case("reactor_200x50")
    w = case.w
    plan = make_plan(api, case, prec)
    p = plan.params_tensor(w.theta)
    d = dev(case.data)
    ref = case.oracle_point(0)
    tol = TOL[prec]
    res = {}
    from paper_1804_07682_gb300 import _native as N
    if prec == "fp64":
        with pytest.raises(N.GnaError):
            plan.tuning = "mapping=slices"
    for m in ("split", "bins") + (("slices",) if prec != "fp64" else ()):
        plan.tuning = f"mapping={m} block=128 nodes=4"
        assert plan.tuning.startswith(f"mapping={m}")
        out = plan.eval(p, d, grad=True, mu=True)
        check_chi2(out["chi2"][0].item(), ref, case.data, w.kind, tol, tag="mapping_choice %s %s" % (prec, m))
        assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < tol
        res[m] = out["chi2"][0].item()
    assert rel(res["split"], res["bins"]) < 2 * tol
    plan.set_graph(True)
    text = plan.autotune(p, d, reps=5)
    assert text.startswith("mapping=")
    out = plan.eval(p, d, grad=True)
    check_chi2(out["chi2"][0].item(), ref, case.data, w.kind, tol, tag="mapping_choice autotuned " + prec)
    plan.close()
    # a plan whose mapping was forced keeps one layout only
    forced = make_plan(api, case, prec, "split")
    from paper_1804_07682_gb300 import _native as N
    with pytest.raises(N.GnaError):
        forced.tuning = "mapping=bins"
    forced.close()


def test_grad_scale_scales_both_arrays_in_place(api):
    # the autograd backward's chain-rule step: a *= s, b *= s in one launch,
    # including a grid-stride pass (more elements than 1024 blocks x 256)
    from paper_1804_07682_gb300 import _native as N
    lib = N.lib()
    s = torch.tensor(-2.5, dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for na, nb in ((4, 0), (0, 7), (4, 1000), (300001, 262145)):
        a = torch.arange(na, dtype=torch.float64, device="cuda") + 0.5
        b = torch.arange(nb, dtype=torch.float64, device="cuda") - 3.0
        a0, b0 = a.clone(), b.clone()
        code = lib.gna_grad_scale(a.data_ptr() if na else None, na, b.data_ptr() if nb else None, nb, s.data_ptr(),
                                  stream)
        assert code == N.GNA_OK
        assert torch.equal(a, a0 * -2.5) and torch.equal(b, b0 * -2.5), (na, nb)


def test_autograd_function(api):
    case = get_case("nuisance_64x1000")
    w = case.w
    plan = make_plan(api, case, "fp64")
    d = dev(case.data)
    theta = dev(w.theta[0]).requires_grad_(True)
    eta = dev(w.eta).requires_grad_(True)
    c = api.chi2(theta, plan, d, eta, w.sigma_eta)
    (2.0 * c).backward(retain_graph=True)
    ref = case.oracle_point(0)
    assert normrel(theta.grad.cpu().numpy(), 2.0 * ref["grad"][:4]) < 1e-9
    assert normrel(eta.grad.cpu().numpy(), 2.0 * ref["grad"][4:]) < 1e-9
    # the kept gradient was handed out (scaled in place): a second backward
    # through the same chi2 is refused, the first one's gradients stay
    with pytest.raises(RuntimeError):
        c.backward()
    assert normrel(theta.grad.cpu().numpy(), 2.0 * ref["grad"][:4]) < 1e-9
    # accumulation over two evaluations
    api.chi2(theta, plan, d, eta, w.sigma_eta).backward()
    assert normrel(theta.grad.cpu().numpy(), 3.0 * ref["grad"][:4]) < 1e-9
    assert normrel(eta.grad.cpu().numpy(), 3.0 * ref["grad"][4:]) < 1e-9
    # first derivatives only: differentiating the gradient again is refused
    (gth,) = torch.autograd.grad(api.chi2(theta, plan, d, eta, w.sigma_eta), theta, create_graph=True)
    assert normrel(gth.detach().cpu().numpy(), ref["grad"][:4]) < 1e-9
    with pytest.raises(RuntimeError):
        gth.sum().backward()

    # FP64 central differences (h = 1e-6 relative) through the same plan
    def f(t):
        with torch.no_grad():
            return api.chi2(dev(t), plan, d, dev(w.eta), w.sigma_eta).item()

    g_fd = oracle.fd_grad(f, w.theta[0])
    assert normrel(ref["grad"][:4], g_fd) < 1e-5

    # a [1, 4] parameter tensor and no nuisances; results of successive calls
    # are independent tensors
    th2 = dev(w.theta[0]).reshape(1, 4).requires_grad_(True)
    c1 = api.chi2(th2, plan, d)
    c2 = api.chi2(dev(w.theta[0] * 1.01), plan, d)
    c1.backward()
    ref0 = oracle.chain(w.edges, w.nodes_per_bin, w.L, w.theta[0], case.N, case.data, w.kind)
    assert c1.dim() == 0 and rel(c1.item(), ref0["chi2"]) < 1e-9 and c2.item() != c1.item()
    assert tuple(th2.grad.shape) == (1, 4) and normrel(th2.grad[0].cpu().numpy(), ref0["grad"][:4]) < 1e-9


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
def test_fits_match_oracle(api, prec):
    case = get_case("fits_8x100x20")
    w = case.w
    plan = make_plan(api, case, prec, per_point_data=True)
    params = plan.params_tensor(w.theta).clone()
    params, chi2 = plan.fit(params, dev(case.data), iters=20, graph=(prec == "ff"))
    torch.cuda.synchronize()
    plan.status()
    P = params.cpu().numpy()
    C = chi2.cpu().numpy()
    for j in range(w.npts):
        ev = lambda t, j=j: oracle.chain(w.edges, w.nodes_per_bin, w.L, t, case.N, case.data[j], w.kind)
        th, c2, _ = oracle.fit_lm(ev, w.theta[j], iters=20)
        pull = float(np.max(np.abs(P[j] - th) / fit_sigma(ev(th))))
        log_err("fit %s" % prec, chi2_rel=rel(C[j], c2), params_rel=rel(P[j], th), pull=pull)
        assert rel(C[j], c2) < (1e-9 if prec == "fp64" else 1e-6), (j, C[j], c2)
        # mixed: largest measured 7.7e-6 relative (5.1e-5 with the double phase)
        assert rel(P[j], th) < (1e-7 if prec == "fp64" else 1e-4), (j, P[j], th)
        # in units of the parameters' statistical errors the two fits agree far
        # inside any physics resolution
        assert pull < (1e-5 if prec == "fp64" else 1e-2), (j, pull)


def test_pseudo_data_matches_oracle_bit_for_bit(api):
    # counter-based draws: the device and the oracle give the same integers
    case = get_case("fits_8x100x20")
    mu = np.concatenate([case.mu_truth, [0.0, 1e-3, 0.7, 699.0, 500.0, 500.001, 12345.6]])
    for seed in (4, 2 ** 40 + 17):
        dev_data = api.poisson_datasets(mu, 300, seed).cpu().numpy()
        ref = oracle.pseudo_data(mu, 300, seed)
        assert np.array_equal(dev_data, ref), seed
    # a prefix does not depend on how many sets one launch draws
    assert np.array_equal(api.poisson_datasets(mu, 40, 4).cpu().numpy(), oracle.pseudo_data(mu, 40, 4))
    from paper_1804_07682_gb300 import _native as N
    with pytest.raises(N.GnaError):
        api.poisson_datasets([1.0, 2e7], 2, 1)
    assert api.poisson_datasets([1.0], 0, 1).numel() == 0


def test_pseudo_data_many_bins_over_several_tables(api):
    # 4000 bins of mean 500 need 20.4 M table entries: the bins are drawn in
    # two ranges of at most 2^24 entries; the draws are the same bit for bit
    rng = np.random.default_rng(8)
    mu = np.full(4000, 500.0)
    mu[::7] = rng.uniform(0.0, 1500.0, mu[::7].size)
    dev_data = api.poisson_datasets(mu, 3, 11).cpu().numpy()
    assert np.array_equal(dev_data, oracle.pseudo_data(mu, 3, 11))


def test_device_status_flags_unphysical_points(api):
    # the parameters live on the device; a point with s2 > 1 is found there
    # and reported by status(), which then clears
    from paper_1804_07682_gb300 import _native as N
    case = get_case("reactor_200x50")
    w = case.w
    plan = make_plan(api, case, "ff")
    d = dev(case.data)
    bad = np.array(w.theta, dtype=np.float64).reshape(1, 4).copy()
    bad[0, 0] = 1.5
    plan.eval(plan.params_tensor(bad), d, grad=True)
    with pytest.raises(N.GnaError):
        plan.status()
    plan.eval(plan.params_tensor(w.theta), d, grad=True)
    plan.status()
    plan.close()


def test_bad_arguments_raise(api):
    from paper_1804_07682_gb300 import _native as N

    case = get_case("reactor_200x50")
    plan = make_plan(api, case, "ff")
    p = plan.params_tensor(case.w.theta)
    with pytest.raises(ValueError):
        plan.eval(p, dev(np.zeros(7)))
    with pytest.raises(N.GnaError):
        plan.fit(p.clone(), dev(np.zeros((1, 200))), iters=0)
    with pytest.raises(N.GnaError):
        plan.tuning = "block=1000"
    with pytest.raises(N.GnaError):
        api.Plan([1.0, 2.0], list(range(1, 18)), nodes_per_bin=4)


# ------------------------------------------------------ any-channel chain --
GEN_TH = np.array([0.307, 0.0218, 0.545, 1.2 * np.pi, 7.53e-5, 2.44e-3])


def general_case(channel, edges, counts, L, npts, e_scale, kind, seed, nuisances=False):
    """Points near GEN_TH, Poisson data from the oracle's prediction at GEN_TH
    (largest node count), normalised to 10^4 events."""
    a, b, anti = channel
    rng = np.random.default_rng(seed)
    theta = np.tile(GEN_TH, (npts, 1)) * rng.uniform(0.97, 1.03, size=(npts, 6))
    counts = np.broadcast_to(np.asarray(counts), (npts,)).astype(np.int32)
    n_t = int(counts.max())
    mu_rb, _ = oracle.binned_general(edges, n_t, L, GEN_TH, a, b, anti, e_scale)
    M = oracle.baseline_weights(np.atleast_1d(L)) @ mu_rb
    N = 1e4 / M.sum()
    data = wl.poisson_data(N * M, seed + 100)
    eta = rng.normal(0.0, 0.02, edges.size - 1) if nuisances else None
    refs = [oracle.chain_general(edges, int(counts[p]), L, theta[p], N, data, a, b, anti, kind, eta,
                                 0.02 if nuisances else 0.0, e_scale) for p in range(npts)]
    return theta, counts, N, data, eta, refs


def check_general(api, channel, prec, edges, counts, L, npts, e_scale, kind, seed, nuisances=False, uniform=True):
    theta, counts, N, data, eta, refs = general_case(channel, edges, counts, L, npts, e_scale, kind, seed, nuisances)
    kw = dict(nodes_per_bin=int(counts[0])) if uniform else dict(node_counts=counts)
    plan = api.Plan(edges, L, npts=npts, norm=N, e_scale=e_scale, prec=prec, kind=KIND_NAMES[kind],
                    channel=channel, **kw)
    out = plan.eval_general(plan.params_tensor(theta), dev(data), None if eta is None else dev(eta),
                            0.02 if nuisances else 0.0, grad=True, grad_eta=nuisances, mu=True)
    torch.cuda.synchronize()
    plan.status()
    # 1e-6 relative on mu in the mixed precisions, also in the bins of a
    # disappearance dip (P ~ 0.01 there; the node pass's cosine sums keep the
    # error relative to P); GNA_FP64: 1e-9 relative, gradient 1e-9
    tol, gtol = (1e-9, 1e-9) if prec == "fp64" else (1e-6, 1e-4)
    tag = "general %s%s%s %s" % (channel[0], channel[1], "bar" if channel[2] else "", prec)
    for p in range(npts):
        ref = refs[p]
        check_chi2(out["chi2"][p].item(), ref, data, kind, tol, tag="%s p%d" % (tag, p))
        mu_err = rel(out["mu"][p].cpu().numpy(), ref["mu"])
        log_err(tag + " mu", mu_rel=mu_err, p_min=float(np.min(ref["mu"] / np.max(ref["mu"]))))
        assert mu_err < tol, (p, mu_err)
        assert normrel(out["grad"][p].cpu().numpy(), ref["grad"][:6]) < gtol, p
        if nuisances:
            assert normrel(out["grad_eta"][p].cpu().numpy(), ref["grad"][6:]) < gtol, p
    plan.close()


KIND_NAMES = {0: "pearson", 1: "poisson"}
CHANNELS = [("mu", "e", False), ("mu", "mu", False), ("mu", "e", True), ("e", "e", True), ("e", "tau", False)]


@pytest.mark.parametrize("channel", CHANNELS)
@pytest.mark.parametrize("prec", ["ff", "f64phase", "fp64"])
def test_general_chain_long_baseline(api, channel, prec):
    # 810 km, 0.5-5 GeV (energies in MeV, spectrum in GeV), 3 points on one
    # grid of 40 bins x 24 nodes: the slice mapping
    check_general(api, channel, prec, np.linspace(500.0, 5000.0, 41), 24, np.array([810.0]), 3, 1e-3, 1, 7)


@pytest.mark.parametrize("L", [[810.0], [810.0, 790.0, 830.0]])
@pytest.mark.parametrize("channel", [("mu", "mu", False), ("mu", "mu", True), ("tau", "tau", False)])
@pytest.mark.parametrize("prec", ["ff", "f64phase", "fp64"])
def test_general_chain_disappearance_dip(api, channel, prec, L):
    # 60 narrow bins of 8 nodes around the first disappearance maximum at
    # 810 km (1.2-2.2 GeV, P down to ~0.01): every bin's mu within 1e-6 of
    # the oracle with no absolute allowance, one and three baselines
    check_general(api, channel, prec, np.linspace(1200.0, 2200.0, 61), 8, np.array(L), 2, 1e-3, 1, 17)


@pytest.mark.parametrize("channel", [("mu", "e", False), ("e", "e", True)])
@pytest.mark.parametrize("prec", ["ff", "fp64"])
def test_general_chain_uneven_grids_baselines_nuisances(api, channel, prec):
    # per-point node counts (two points share one), three baselines (four-baseline
    # kernel with a zero-weight slot), Pearson chi^2 with nuisances: the bin mapping
    check_general(api, channel, prec, np.linspace(500.0, 5000.0, 71), [12, 30, 12, 7], np.array([810.0, 295.0, 1300.0]),
                  4, 1e-3, 0, 9, nuisances=True, uniform=False)


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("prec", ["ff", "fp64"])
def test_general_chain_sparse_counts(api, prec, kind):
    # 200 nu_mu -> nu_e events over 40 bins: Poisson data with empty bins
    # (the d = 0 terms of both chi^2 kinds) and mu of a few events per bin
    edges = np.linspace(500.0, 5000.0, 41)
    n, L = 16, np.array([810.0])
    mu_rb, _ = oracle.binned_general(edges, n, L, GEN_TH, "mu", "e", False, 1e-3)
    N = 200.0 / mu_rb[0].sum()
    data = wl.poisson_data(N * mu_rb[0], 123)
    assert np.any(data == 0)
    theta = GEN_TH * np.array([1.02, 0.98, 1.01, 0.97, 1.03, 0.99])
    ref = oracle.chain_general(edges, n, L, theta, N, data, "mu", "e", False, kind, None, 0.0, 1e-3)
    plan = api.Plan(edges, L, nodes_per_bin=n, norm=N, e_scale=1e-3, prec=prec, kind=KIND_NAMES[kind],
                    channel=("mu", "e", False))
    out = plan.eval_general(plan.params_tensor(theta[None, :]), dev(data), grad=True, mu=True)
    torch.cuda.synchronize()
    plan.status()
    tol, gtol = (1e-9, 1e-9) if prec == "fp64" else (1e-6, 1e-4)
    check_chi2(out["chi2"][0].item(), ref, data, kind, tol, tag="general sparse %s %d" % (prec, kind))
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < tol
    assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:6]) < gtol
    plan.close()


@pytest.mark.parametrize("prec", ["ff", "fp64"])
def test_general_chain_boundary_parameters(api, prec):
    # any-channel coefficients next to the edges of the domain (a plan
    # reports a sin^2 at exactly 0 or 1 as outside it: the mixing matrix
    # holds square roots, whose derivatives diverge there): theta13 -> 0,
    # theta23 -> 0 and 90 degrees, theta12 -> 90 degrees, and the
    # CP-conserving delta = 0 and pi; nu_mu -> nu_e at 810 km
    edges = np.linspace(500.0, 5000.0, 41)
    n, L = 16, np.array([810.0])
    g, e = GEN_TH, 1e-10
    theta = np.array([[g[0], e, g[2], g[3], g[4], g[5]], [g[0], g[1], e, g[3], g[4], g[5]],
                      [g[0], g[1], 1.0 - e, g[3], g[4], g[5]], [g[0], g[1], g[2], 0.0, g[4], g[5]],
                      [1.0 - e, g[1], g[2], g[3], g[4], g[5]], [g[0], g[1], g[2], np.pi, g[4], g[5]]])
    mu_rb, _ = oracle.binned_general(edges, n, L, GEN_TH, "mu", "e", False, 1e-3)
    N = 1e4 / mu_rb[0].sum()
    data = wl.poisson_data(N * mu_rb[0], 5)
    plan = api.Plan(edges, L, npts=theta.shape[0], nodes_per_bin=n, norm=N, e_scale=1e-3, prec=prec, kind="poisson",
                    channel=("mu", "e", False))
    out = plan.eval_general(plan.params_tensor(theta), dev(data), grad=True, mu=True)
    torch.cuda.synchronize()
    plan.status()
    tol, gtol = (1e-9, 1e-9) if prec == "fp64" else (1e-6, 1e-4)
    for p in range(theta.shape[0]):
        ref = oracle.chain_general(edges, n, L, theta[p], N, data, "mu", "e", False, 1, None, 0.0, 1e-3)
        check_chi2(out["chi2"][p].item(), ref, data, 1, tol, tag="general boundary %s p%d" % (prec, p))
        assert rel(out["mu"][p].cpu().numpy(), ref["mu"]) < tol, p
        assert normrel(out["grad"][p].cpu().numpy(), ref["grad"][:6]) < gtol, p
    plan.close()


@pytest.mark.parametrize("mapping", [None, "bins"])
def test_general_repeated_evaluations_are_bit_identical(api, mapping):
    # the any-channel chain's sums (node, slice, group, point) also run in a
    # fixed order: repeated evaluations agree bit for bit
    theta, counts, N, data, eta, refs = general_case(("mu", "e", False), np.linspace(500.0, 5000.0, 41), 64,
                                                     np.array([810.0, 790.0]), 3, 1e-3, 1, 21)
    plan = api.Plan(np.linspace(500.0, 5000.0, 41), [810.0, 790.0], npts=3, nodes_per_bin=64, norm=N, e_scale=1e-3,
                    prec="ff", kind="poisson", channel=("mu", "e", False), mapping=mapping)
    p, d = plan.params_tensor(theta), dev(data)
    outs = [{k: v.clone() for k, v in plan.eval_general(p, d, grad=True, mu=True).items()} for _ in range(5)]
    for o in outs[1:]:
        for k in o:
            assert torch.equal(o[k], outs[0][k]), k
    plan.close()


def test_general_chain_reactor_many_nodes(api):
    # nue_bar survival through the any-channel chain on a reactor-like grid of
    # 20 bins x 2048 nodes and eight baselines (slices of the nodes)
    check_general(api, ("e", "e", True), "ff", np.linspace(1.8, 9.0, 21), 2048,
                  np.array([52.5, 52.8, 53.0, 52.2, 1.6, 1.9, 5.0, 40.0]), 1, 1.0, 1, 11)


def test_general_plan_calls_and_status(api):
    edges = np.linspace(500.0, 5000.0, 11)
    gp = api.Plan(edges, [810.0], nodes_per_bin=8, e_scale=1e-3, channel=("mu", "e", False))
    d = torch.full((10,), 50.0, dtype=torch.float64, device="cuda")
    from paper_1804_07682_gb300 import _native as N
    with pytest.raises(N.GnaError):  # the survival-chain call on an any-channel plan
        gp.eval(torch.zeros(1, 4, dtype=torch.float64, device="cuda"), d)
    ep = api.Plan(edges, [810.0], nodes_per_bin=8, e_scale=1e-3)
    with pytest.raises(ValueError):
        ep.eval_general(torch.zeros(1, 6, dtype=torch.float64, device="cuda"), d)
    ep.close()
    # a mixing parameter on the boundary is reported by status()
    bad = GEN_TH.copy()
    bad[2] = 0.0
    gp.eval_general(gp.params_tensor(bad), d)
    torch.cuda.synchronize()
    with pytest.raises(N.GnaError):
        gp.status()
    gp.eval_general(gp.params_tensor(GEN_TH), d)
    torch.cuda.synchronize()
    gp.status()
    # the autotuner times block sizes and slice lengths of the plan's mapping
    tuning = gp.autotune(gp.params_tensor(GEN_TH), d, reps=1)
    assert tuning.startswith("mapping=slices")
    r = gp.eval_general(gp.params_tensor(GEN_TH), d, mu=True)
    ref = oracle.chain_general(edges, 8, [810.0], GEN_TH, 1.0, d.cpu().numpy(), "mu", "e", kind=0, e_scale=1e-3)
    assert rel(r["chi2"][0].item(), ref["chi2"]) < 1e-6
    gp.close()


@pytest.mark.parametrize("prec", ["ff", "f64phase", "fp64"])
def test_general_chain_per_point_data_and_chi2_only(api, prec):
    # one data row per point, and chi^2 alone (no gradient: six node sums per
    # bin instead of twelve), through the slice mapping
    channel = ("mu", "e", False)
    edges = np.linspace(500.0, 5000.0, 37)
    theta, counts, N, data, eta, refs = general_case(channel, edges, 40, np.array([810.0]), 3, 1e-3, 1, 21)
    rows = np.stack([wl.poisson_data(refs[p]["mu"], 30 + p) for p in range(3)])
    plan = api.Plan(edges, [810.0], nodes_per_bin=40, npts=3, norm=N, e_scale=1e-3, prec=prec, kind="poisson",
                    max_datasets=3, channel=channel)
    out = plan.eval_general(plan.params_tensor(theta), dev(rows), grad=False, mu=True)
    torch.cuda.synchronize()
    plan.status()
    assert "grad" not in out
    for p in range(3):
        ref = oracle.chain_general(edges, 40, [810.0], theta[p], N, rows[p], "mu", "e", False, 1, e_scale=1e-3)
        check_chi2(out["chi2"][p].item(), ref, rows[p], 1, TOL[prec], tag="general rows %s p%d" % (prec, p))
        assert rel(out["mu"][p].cpu().numpy(), ref["mu"]) < 1e-6, p
    plan.close()


def test_general_chain_through_autograd(api):
    # the autograd Function on an any-channel plan (GNA_FP64): the gradient in
    # the six parameters and the nuisances against the oracle
    channel = ("mu", "e", True)
    edges = np.linspace(500.0, 5000.0, 25)
    theta, counts, N, data, eta, refs = general_case(channel, edges, 16, np.array([810.0]), 1, 1e-3, 1, 41,
                                                     nuisances=True)
    plan = api.Plan(edges, [810.0], nodes_per_bin=16, norm=N, e_scale=1e-3, prec="fp64", kind="poisson",
                    channel=channel)
    th = dev(theta[0]).requires_grad_(True)
    et = dev(eta).requires_grad_(True)
    c = api.chi2(th, plan, dev(data), et, 0.02)
    (3.0 * c).backward()
    ref = refs[0]
    assert rel(c.item(), ref["chi2"]) < 1e-9
    assert normrel(th.grad.cpu().numpy(), 3.0 * ref["grad"][:6]) < 1e-9
    assert normrel(et.grad.cpu().numpy(), 3.0 * ref["grad"][6:]) < 1e-9
    plan.close()


@pytest.mark.parametrize("graph", [False, True])
def test_general_chain_from_host_buffers(api, graph):
    # the any-channel chain from host buffers (one packed copy in, one out):
    # the device call's results bit for bit, two evaluations in flight, and
    # the survival chain's host calls refuse the plan
    from paper_1804_07682_gb300 import _native as N
    channel = ("mu", "e", False)
    edges = np.linspace(500.0, 5000.0, 31)
    theta, counts, Nn, data, eta, refs = general_case(channel, edges, 16, np.array([810.0]), 3, 1e-3, 1, 51,
                                                      nuisances=True)
    plan = api.Plan(edges, [810.0], nodes_per_bin=16, npts=3, norm=Nn, e_scale=1e-3, prec="ff", kind="poisson",
                    channel=channel)
    plan.set_graph(graph)
    d_out = plan.eval_general(plan.params_tensor(theta), dev(data), dev(eta), 0.02, grad=True)
    torch.cuda.synchronize()
    c, g = plan.eval_host(theta, data, eta, 0.02, grad=True)
    assert np.array_equal(c, d_out["chi2"].cpu().numpy()) and np.array_equal(g, d_out["grad"].cpu().numpy())
    th1 = theta * np.array([1.01, 0.99, 1.02, 0.98, 1.0, 1.01])
    for _ in range(2):
        t0 = plan.eval_host_async(theta, data, eta, 0.02)
        t1 = plan.eval_host_async(th1, data, eta, 0.02)
        c0, g0 = plan.eval_host_wait(t0)
        c1, g1 = plan.eval_host_wait(t1)
        assert np.array_equal(c0, c) and np.array_equal(g0, g)
    for p in range(3):
        check_chi2(c[p], refs[p], data, 1, 1e-6, tag="general host p%d" % p)
        assert normrel(g[p], refs[p]["grad"][:6]) < 1e-4
        r1 = oracle.chain_general(edges, 16, [810.0], th1[p], Nn, data, "mu", "e", False, 1, eta, 0.02, e_scale=1e-3)
        check_chi2(c1[p], r1, data, 1, 1e-6, tag="general host th1 p%d" % p)
    code = N.lib().gna_chain_eval_host(plan._h, ctypes.c_void_p(theta.ctypes.data), None, 0.0,
                                       ctypes.c_void_p(data.ctypes.data), 0, ctypes.c_void_p(c.ctypes.data), None, None,
                                       None)
    assert code == N.GNA_ESTATE
    plan.close()


@pytest.mark.parametrize("prec", ["fp64", "ff"])
def test_general_fits_match_oracle(api, prec):
    # batched Levenberg-Marquardt fits in all six parameters of nu_mu -> nu_e
    # appearance at 810 km (40 bins x 12 nodes, 0.5-5 GeV): 6 Poisson
    # pseudo-data sets from the oracle's prediction at GEN_TH, starts
    # perturbed by up to 3 %; each fitted again by the oracle's fit_lm
    edges = np.linspace(500.0, 5000.0, 41)
    n, k = 12, 6
    mu_rb, _ = oracle.binned_general(edges, n, [810.0], GEN_TH, "mu", "e", False, 1e-3)
    Nn = 2e4 / mu_rb[0].sum()
    data = np.stack([wl.poisson_data(Nn * mu_rb[0], 70 + j) for j in range(k)])
    start = np.tile(GEN_TH, (k, 1)) * np.random.default_rng(61).uniform(0.97, 1.03, size=(k, 6))
    plan = api.Plan(edges, [810.0], nodes_per_bin=n, npts=k, norm=Nn, e_scale=1e-3, prec=prec, kind="poisson",
                    max_datasets=k, channel=("mu", "e", False))
    params = plan.params_tensor(start).clone()
    params, chi2 = plan.fit(params, dev(data), iters=20, graph=(prec == "ff"))
    torch.cuda.synchronize()
    plan.status()
    P, C = params.cpu().numpy(), chi2.cpu().numpy()
    start_chi2 = [oracle.chain_general(edges, n, [810.0], start[j], Nn, data[j], "mu", "e", False, 1,
                                       e_scale=1e-3)["chi2"] for j in range(k)]
    for j in range(k):
        ev = lambda t, j=j: oracle.chain_general(edges, n, [810.0], t, Nn, data[j], "mu", "e", False, 1, e_scale=1e-3)
        th, c2, _ = oracle.fit_lm(ev, start[j], iters=20)
        log_err("general fit %s" % prec, chi2_rel=rel(C[j], c2), params_rel=rel(P[j], th))
        assert C[j] <= start_chi2[j] * (1 + 1e-12)
        assert rel(C[j], c2) < (1e-9 if prec == "fp64" else 1e-6), (j, C[j], c2)
        # mixed: up to 5.4e-4 relative measured.  One appearance channel does
        # not determine six parameters (the Fisher matrix's condition number
        # is ~3e17 at the generating point), so the fits wander along flat
        # directions and no statistical errors exist to measure them in
        assert rel(P[j], th) < (1e-7 if prec == "fp64" else 1e-3), (j, P[j], th)
    plan.close()


# ------------------------------------------- chunk-anchored node kernels
@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("mapping", ["bins", "slices"])
@pytest.mark.parametrize("nL", [1, 2, 3, 5, 9])
@pytest.mark.parametrize("inverted", [False, True])
@pytest.mark.parametrize("n,edges", [(1, (2.0, 9.0)), (3, (2.0, 9.0)), (4, (2.0, 9.0)), (5, (3.0, 3.4)), (33, (3.0, 3.4)),
                                     (130, (3.0, 3.4)), (67, (0.6, 12.0))])
def test_anchored_chunks(api, prec, mapping, nL, n, edges, inverted):
    # orders around a quad and a chunk of nodes; fine grids (3-3.4 MeV: long
    # chunks), coarse ones (2-9 MeV with up to 5 nodes: every phase reduced)
    # and one that has both and lengths between (0.6-12 MeV); baselines below,
    # at and beyond the packed instantiations; 37 bins: a ragged group; either
    # mass ordering (a negative dm2_32: negative quotients of the phases)
    rng = np.random.default_rng(nL + n)
    e = np.linspace(edges[0], edges[1], 38)
    L = rng.uniform(1.0, 60.0, nL)
    theta = np.array(wl.TRUTH) * 1.03 * ([1, 1, 1, -1] if inverted else 1)
    Nn = oracle.norm_for_total(e, n, L, wl.TRUTH)
    data = wl.poisson_data(Nn * (oracle.baseline_weights(L) @ oracle.binned(e, n, L, wl.TRUTH)), 7)
    ref = oracle.chain(e, n, L, theta, Nn, data, wl.POISSON)
    plan = api.Plan(e, L, nodes_per_bin=n, norm=Nn, prec=prec, kind="poisson", mapping=mapping)
    if mapping == "slices":
        plan.tuning = "slice=16"
    p, d = plan.params_tensor(theta), dev(data)
    out = plan.eval(p, d, grad=True, mu=True, spectra=True)
    alone = plan.eval(p, d, grad=False)
    torch.cuda.synchronize()
    plan.status()
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < 1e-6
    assert rel(out["spectra"][0].cpu().numpy(), ref["mu_rb"]) < 1e-6
    assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:4]) < 1e-4
    for o in (out, alone):  # few nodes per bin: the scaled bound (see the module's head)
        check_chi2(o["chi2"][0].item(), ref, data, wl.POISSON, 1e-6, tag="anchored %d %d" % (nL, n), plain=False)
    plan.close()


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("nL", [1, 2, 3, 5])
@pytest.mark.parametrize("channel", [("mu", "e", False), ("mu", "mu", True), ("e", "tau", False)])
@pytest.mark.parametrize("inverted", [False, True])
@pytest.mark.parametrize("n,edges", [(1, (600.0, 4000.0)), (3, (600.0, 4000.0)), (5, (1500.0, 2000.0)), (34, (1500.0, 2000.0)),
                                     (131, (1500.0, 2000.0)), (21, (150.0, 3000.0))])
def test_general_anchored_chunks(api, prec, nL, channel, n, edges, inverted):
    # as test_anchored_chunks for the any-channel node kernels: single nodes,
    # quads, chunks and ragged ends, coarse and fine grids, both mappings and orderings
    rng = np.random.default_rng(nL + n)
    e = np.linspace(edges[0], edges[1], 38)
    L = np.array([810.0, 295.0, 735.0, 700.0, 280.0])[:nL]
    th = np.array(THETA_FULL) * 1.02 * ([1, 1, 1, 1, 1, -1] if inverted else 1)
    a, b, anti = channel
    mu_rb, _ = oracle.binned_general(e, n, L, THETA_FULL, a, b, anti, 1e-3)
    M = oracle.baseline_weights(L) @ mu_rb
    Nn = 1e4 / M.sum()
    data = wl.poisson_data(Nn * M, 3)
    ref = oracle.chain_general(e, n, L, th, Nn, data, a, b, anti, 1, None, 0.0, 1e-3)
    for mapping in ("bins", "slices"):
        plan = api.Plan(e, L, nodes_per_bin=n, norm=Nn, e_scale=1e-3, prec=prec, kind="poisson", channel=channel,
                        mapping="bins" if mapping == "bins" else None)
        if mapping == "slices":
            plan.tuning = "slice=16"
        p, d = plan.params_tensor(th), dev(data)
        out = plan.eval_general(p, d, grad=True, mu=True)
        alone = plan.eval_general(p, d, grad=False)
        torch.cuda.synchronize()
        plan.status()
        assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < 1e-6
        assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:6]) < 1e-4
        for o in (out, alone):
            check_chi2(o["chi2"][0].item(), ref, data, wl.POISSON, 1e-6, tag="general anchored %d %d" % (nL, n), plain=False)
        plan.close()


@pytest.mark.parametrize("nL", [1, 3, 9])
@pytest.mark.parametrize("inverted", [False, True])
@pytest.mark.parametrize("n,edges", [(1, (2.0, 9.0)), (3, (2.0, 9.0)), (5, (3.0, 3.4)), (33, (3.0, 3.4)), (130, (3.0, 3.4)),
                                     (1000, (3.0, 3.4)), (67, (0.6, 12.0))])
def test_fp64_anchored_chunks(api, nL, n, edges, inverted):
    # GNA_FP64: sincos per node (coarse grids), both lengths of polynomial
    # (0.6-12 MeV has all three), whole bins and slices, both mass orderings
    rng = np.random.default_rng(nL + n)
    e = np.linspace(edges[0], edges[1], 38)
    L = rng.uniform(1.0, 60.0, nL)
    theta = np.array(wl.TRUTH) * 1.03 * ([1, 1, 1, -1] if inverted else 1)
    Nn = oracle.norm_for_total(e, n, L, wl.TRUTH)
    data = wl.poisson_data(Nn * (oracle.baseline_weights(L) @ oracle.binned(e, n, L, wl.TRUTH)), 7)
    ref = oracle.chain(e, n, L, theta, Nn, data, wl.POISSON)
    for npts in (1, 40):
        plan = api.Plan(e, L, nodes_per_bin=n, npts=npts, norm=Nn, prec="fp64", kind="poisson")
        p, d = plan.params_tensor(np.repeat(theta[None], npts, 0)), dev(data)
        out = plan.eval(p, d, grad=True, mu=True, spectra=True)
        alone = plan.eval(p, d, grad=False)
        torch.cuda.synchronize()
        plan.status()
        q = npts - 1
        assert rel(out["mu"][q].cpu().numpy(), ref["mu"]) < 1e-9
        assert rel(out["spectra"][q].cpu().numpy(), ref["mu_rb"]) < 1e-9
        assert normrel(out["grad"][q].cpu().numpy(), ref["grad"][:4]) < 1e-9
        for o in (out, alone):
            check_chi2(o["chi2"][q].item(), ref, data, wl.POISSON, 1e-9, tag="fp64 anchored %d %d" % (nL, n), plain=False)
        plan.close()


@pytest.mark.parametrize("nL", [1, 3])
@pytest.mark.parametrize("channel", [("mu", "e", False), ("mu", "mu", True)])
@pytest.mark.parametrize("inverted", [False, True])
@pytest.mark.parametrize("n,edges", [(1, (600.0, 4000.0)), (5, (1500.0, 2000.0)), (131, (1500.0, 2000.0)), (21, (150.0, 3000.0))])
def test_fp64_general_anchored_chunks(api, nL, channel, n, edges, inverted):
    e = np.linspace(edges[0], edges[1], 38)
    L = np.array([810.0, 295.0, 735.0])[:nL]
    th = np.array(THETA_FULL) * 1.02 * ([1, 1, 1, 1, 1, -1] if inverted else 1)
    a, b, anti = channel
    mu_rb, _ = oracle.binned_general(e, n, L, THETA_FULL, a, b, anti, 1e-3)
    M = oracle.baseline_weights(L) @ mu_rb
    Nn = 1e4 / M.sum()
    data = wl.poisson_data(Nn * M, 3)
    ref = oracle.chain_general(e, n, L, th, Nn, data, a, b, anti, 1, None, 0.0, 1e-3)
    plan = api.Plan(e, L, nodes_per_bin=n, norm=Nn, e_scale=1e-3, prec="fp64", kind="poisson", channel=channel)
    p, d = plan.params_tensor(th), dev(data)
    out = plan.eval_general(p, d, grad=True, mu=True)
    alone = plan.eval_general(p, d, grad=False)
    torch.cuda.synchronize()
    plan.status()
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < 1e-9
    assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:6]) < 1e-9
    for o in (out, alone):
        check_chi2(o["chi2"][0].item(), ref, data, wl.POISSON, 1e-9, tag="fp64 general %d %d" % (nL, n), plain=False)
    plan.close()


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
@pytest.mark.parametrize("inverted", [False, True])
def test_oscprob_number_ranges(api, prec, inverted):
    """Energies at the edges of the number range, and phases from next to zero
    to many turns, in both mass orderings: each against the formula in double."""
    E = np.array([5.0, 1.0, 2.0, np.nextafter(2.0, 0.0), np.nextafter(1.0, 2.0), 2.0 ** -20, 2.0 ** 20, 3e9, 1e15, 1e30,
                  1e300, 2.0 ** -1000, -5.0, np.inf, np.nan])
    L = [0.0, 52.5, 1.7, 1e4]
    for channel in (None, ("mu", "e"), ("mu", "mu")):
        th = THETA_FULL[:5] + (-THETA_FULL[5] if inverted else THETA_FULL[5],)
        if channel is None:
            P = api.oscprob(dev(E), L, [th[i] for i in (0, 1, 4, 5)], prec).double().cpu().numpy()
        else:
            P = api.oscprob_general(dev(E), L, th, *channel, prec=prec).double().cpu().numpy()
        with np.errstate(all="ignore"):
            ref = np.array([oracle_prob(*(channel or ("e", "e")), E, Lr, False, th) for Lr in L])
            phase = np.array([1266.932679419849 * Lr * (th[4] + abs(th[5])) / np.abs(E) for Lr in L])
        # double: the phase's rounding, twice its 2^-53; mixed: FP32 polynomials
        # (2e-7 each) and, in double-float, 2^-44 of the phase up to its 2^12 pi
        top = {"fp64": 1e9, "f64phase": 1e6, "ff": 1e4}[prec]
        ok = np.isfinite(ref) & (phase < top)
        if prec != "fp64":  # 1/E is a pair of floats
            ok &= (np.abs(E) < 1e18) & (np.abs(E) > 1e-18)
        tol = {"fp64": 4e-16 + 1e-15 * phase, "f64phase": 6e-7 + 1e-12 * phase, "ff": 6e-7 + 1e-11 * phase}[prec]
        # compared: every energy of 1 - 5 MeV at 52.5 and 1.7 km, and no phase at all (0 km)
        assert ok[:3, :5].all()
        assert (np.abs(P - ref)[ok] <= tol[ok]).all()
        if prec == "fp64":
            # probabilities next to zero or one: the terms (up to 2x each) are
            # good to 2^-53 of themselves
            small = ok & (phase < 1e-2)
            assert (np.abs(P - ref)[small] <= 1e-15 * phase[small] + (3e-16 if channel != ("mu", "e") else 0)).all()
            assert np.isnan(P[1:, -1]).all()


@pytest.mark.parametrize("nL", [2, 5, 6, 9, 12, 16])
@pytest.mark.parametrize("nodes", [3, 10, 50, 129])
def test_baseline_groups_and_short_slices(api, nL, nodes):
    """Baselines taken 2, 4, 6 or 8 at a time in one or two passes, and slices
    down to one quad of nodes, against the kernel-per-step FP64 chain."""
    rng = np.random.default_rng(nL * 100 + nodes)
    edges = np.linspace(1.8, 8.0, 71)
    L = list(rng.uniform(1.0, 60.0, nL))
    th = np.array([[0.307, 0.0218, 7.53e-5, 2.44e-3]])
    plain = api.Plan(edges, L, nodes_per_bin=nodes, prec="fp64", kind="poisson", with_plain=True)
    ref0 = plain.eval(plain.params_tensor(th), dev(np.full(70, 1.0)), grad=True, spectra=True, mu=True)
    data = dev(rng.poisson(1e4 * ref0["mu"].cpu().numpy().ravel() / ref0["mu"].max().item()) * 1.0)
    norm = 1e4 / ref0["mu"].max().item()
    out = {}
    for prec in ("fp64", "ff"):
        plan = api.Plan(edges, L, nodes_per_bin=nodes, prec=prec, kind="poisson", norm=norm, with_plain=prec == "fp64")
        out[prec] = plan.eval(plan.params_tensor(th), data, grad=True, spectra=True, plain=prec == "fp64")
        chi_only = plan.eval(plan.params_tensor(th), data)["chi2"]
        assert rel(chi_only.cpu().numpy(), out[prec]["chi2"].cpu().numpy()) < 1e-6
    a, b = out["ff"], out["fp64"]
    assert rel(a["spectra"].cpu().numpy(), b["spectra"].cpu().numpy()) < 1e-6
    # chi^2 within 1e-6 of what a relative change of every mu_i makes of it
    scale = max(b["chi2"].item(), 2 * float(torch.sqrt(data).sum()))
    assert abs(a["chi2"].item() - b["chi2"].item()) < 1e-6 * scale
    assert normrel(a["grad"].cpu().numpy(), b["grad"].cpu().numpy()) < 1e-4


@pytest.mark.parametrize("nbins,n", [(200, 50), (40, 1031)])
def test_fp64_fits_keep_their_mapping_through_tuning(api, nbins, n):
    """The fits of a default GNA_FP64 plan run in the split mapping while its
    evaluations go by bins: reading the tuning and setting it back, and
    autotuning the evaluations, change no bit of a fit."""
    edges, L = np.linspace(1.8, 8.0, nbins + 1), [52.5, 30.0]
    th = np.array(wl.TRUTH)
    Nn = oracle.norm_for_total(edges, n, L, wl.TRUTH)
    data = dev(wl.pseudo_datasets(Nn * (oracle.baseline_weights(L) @ oracle.binned(edges, n, L, wl.TRUTH)), 2, 5))
    plan = api.Plan(edges, L, nodes_per_bin=n, npts=2, norm=Nn, prec="fp64", kind="poisson", max_datasets=2)

    def fit():
        p, c = plan.fit(plan.params_tensor(np.repeat(1.02 * th[None], 2, 0)), data, iters=6)
        return np.concatenate([p.cpu().numpy().ravel(), c.cpu().numpy()])

    first = fit()
    plan.tuning = plan.tuning
    assert np.array_equal(first, fit())
    assert plan.tuning.startswith("mapping=bins") and plan.tuning.endswith("fit=split")
    if plan.autotune(plan.params_tensor(np.repeat(th[None], 2, 0)), data[0].contiguous(), reps=2).startswith("mapping=bins"):
        assert np.array_equal(first, fit())
    plan.tuning = "mapping=split block=256 nodes=16"  # named: evaluations and fits
    assert np.array_equal(first, fit())
    plan.tuning = "mapping=bins"
    assert "fit" not in plan.tuning
    by_bins = fit()
    assert rel(by_bins, first) < 1e-6
    plan.tuning = "fit=split"
    assert np.array_equal(first, fit())
    with pytest.raises(N.GnaError):
        plan.tuning = "fit=slices"
    plan.close()


def test_oscprob_fp64_next_to_its_zeros(api):
    """P(mu -> e) with dm2_21 = 0 vanishes where x32 is a multiple of pi, and
    the survival probability at maximal mixing where x21 is an odd multiple of
    pi / 2: P stays at or above zero there and follows the closed form."""
    ld = np.longdouble
    K = ld(10) ** 3 / (4 * ld("0.1973269804"))
    rng = np.random.default_rng(8)
    off = np.concatenate([10.0 ** rng.uniform(-12, -0.5, 20000), [0.0]]) * rng.choice([-1.0, 1.0], 20001)
    pi = ld("3.14159265358979323846264338327950288")
    for form, x0, L in (("mu-e", pi, 810.0), ("mu-e", 7 * pi, 1300.0), ("max", pi / 2, 52.5), ("max", 7 * pi / 2, 180.0)):
        c = K * (ld(2.44e-3) if form == "mu-e" else ld(7.53e-5)) * ld(L)
        E = (c / (x0 + off)).astype(np.float64)
        if form == "mu-e":
            s13, s23 = 0.0218, 0.545
            P = api.oscprob_general(dev(E), [L], (0.307, s13, s23, 0.7, 0.0, 2.44e-3), "mu", "e", prec="fp64")
            A, x = 4 * ld(s23) * ld(s13) * (1 - ld(s13)), c / E.astype(ld)
        else:
            P = api.oscprob(dev(E), [L], (0.5, 0.0, 7.53e-5, 0.0), "fp64")
            A, x = ld(1), c / E.astype(ld) - pi / 2
        P, s = P[0].cpu().numpy(), np.abs(np.sin(x))
        ref = A * s * s
        # the phase is good to 4 roundings of 2^-53, in the closed form and the
        # library's constants; the sum of up to three terms to 2^-50 of itself
        dx = 4 * 2.0 ** -53 * float(x0)
        tol = A * (2 * s * dx + dx * dx) + 2.0 ** -50 * ref
        if form == "max":  # one minus a square: 2^-52 of one
            tol = tol + 2.0 ** -52
        assert (P >= 0).all(), (form, float(x0), P.min())
        assert (np.abs(P - ref) <= tol).all(), (form, float(x0), float((np.abs(P - ref) / tol).max()))


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("nL", [1, 2])
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("n", [7, 64, 129])
def test_chunk_weights_where_p_vanishes(api, general, nL, prec, n):
    """Maximal two-flavour mixing at an oscillation minimum: P is the square of
    a small angle, and the prediction what is left of the bin's weight when the
    chunks' weights are taken from it: their sums hold to 2^-38 of the weight."""
    K = 1e3 / (4 * 0.1973269804)
    L, dm = 52.5, 7.53e-5
    E0 = K * dm * L / (np.pi / 2)
    e = np.linspace(E0 * (1 - 1e-5), E0 * (1 + 1e-5), 34)
    mid = 0.5 * (e[1:] + e[:-1])
    if general:  # nu_e survival of the any-channel chain (mixing inside (0, 1))
        th, kw = [0.5, 1e-15, 0.5, 0.3, dm, 1e-12], dict(channel=("e", "e", False))
    else:
        th, kw = [0.5, 0.0, dm, 0.0], {}
    plan = api.Plan(e, [L] * nL, nodes_per_bin=n, prec=prec, kind="poisson", **kw)
    p, d = plan.params_tensor(th), dev(np.ones(33))
    mu = (plan.eval_general if general else plan.eval)(p, d, grad=True, mu=True)["mu"][0].cpu().numpy()
    plan.status()
    plan.close()
    W = np.exp(0.87 - 0.16 * mid - 0.091 * mid * mid) * np.diff(e)
    x = K * dm * L / np.linspace(e[:-1], e[1:], 33)
    ref = W * (np.cos(x) ** 2).mean(axis=0)  # P <= 2.5e-10
    # 2^-38 of the weight from the sums; the reduced phase of pi holds to 2^-24
    # of the largest offset, 1.6e-5 (its square to 2^-23)
    assert (np.abs(mu - ref) <= W * (2.0 ** -38 + 2.0 ** -22 * 2.5e-10)).all(), float((np.abs(mu - ref) / W).max())


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("channel", [None, ("mu", "mu", False)])
@pytest.mark.parametrize("mapping", ["bins", "slices"])
@pytest.mark.parametrize("norm,top", [(1e60, 15.0), (1e-30, 15.0), (1e-44, 15.0), (1e-60, 15.0), (1e-20, 30.0), (1e33, 36.0)])
def test_normalisations_of_any_size(api, prec, channel, mapping, norm, top):
    """Normalisations and predictions outside the range of a float: the
    prediction scales with the normalisation (up to 36 MeV the spectrum falls
    by 45 orders of magnitude), and so do the derivatives by the nuisances
    where the prediction is a float (their residual is one)."""
    e = np.linspace(1.8, top, 41)
    L, th = [52.5, 30.0], [0.307, 0.0218, 7.53e-5, 2.44e-3]
    if channel:
        th = [0.307, 0.0218, 0.545, 0.7, 7.53e-5, 2.44e-3]
    out = {}
    for N_, pr in ((1.0, "fp64"), (norm, prec)):
        plan = api.Plan(e, L, nodes_per_bin=20, norm=N_, prec=pr, kind="poisson", channel=channel,
                        mapping=None if pr == "fp64" or (channel and mapping == "slices") else mapping)
        f = plan.eval if channel is None else plan.eval_general
        o = f(plan.params_tensor(th), dev(np.zeros(40)), eta=dev(np.linspace(-0.5, 1.0, 40)), sigma=0.0, grad=True,
              grad_eta=True, mu=True)
        out[pr] = o["mu"][0].cpu().numpy(), o["grad_eta"][0].cpu().numpy()
        plan.status()
        plan.close()
    ref, got = out["fp64"], out[prec]
    # weights are FP32: below 2^-126 they keep 2^-149 of one each (2 MeV wide bins, 20 nodes)
    low = 20 * 2.0 ** -149
    a_float = (ref[0] * norm > 1e-37) & (ref[0] * norm < 1e38) & (ref[0] > 1e-37)
    for a, b, ok in zip(got, ref, (np.ones(40, bool), a_float)):
        assert (np.abs(a / norm - b) <= 2e-6 * np.abs(b) + 4 * low)[ok].all(), (a / norm, b)


def derivative_errors(api, e, L, n, prec, channel=None, e_scale=1.0, seed=1):
    """rms over 64 points of the errors of mu and of its derivatives by the
    parameters, one bin, in units of their own rms: Pearson's chi^2 of no
    counts is mu, so its gradient is d mu.  Against GNA_FP64."""
    rng = np.random.default_rng(seed)
    th = np.array(THETA_FULL) * (1 + rng.uniform(-0.05, 0.05, (64, 6)))
    if channel is None:
        th = th[:, [0, 1, 4, 5]]
    out = []
    for p in (prec, "fp64"):
        plan = api.Plan(e, L, nodes_per_bin=n, npts=64, prec=p, kind="pearson", channel=channel, e_scale=e_scale)
        o = (plan.eval if channel is None else plan.eval_general)(plan.params_tensor(th), dev(np.zeros(1)), grad=True, mu=True)
        out.append(np.concatenate([o["mu"].cpu().numpy(), o["grad"].cpu().numpy()], axis=1))
        plan.close()
    a, b = out
    return np.sqrt(((a - b) ** 2).mean(axis=0) / (b ** 2).mean(axis=0))


def s12_cancellation(e, L, seed=1):
    """Over derivative_errors' points: rms of the absolute terms of d mu / d
    s2_12 over rms of their sum (survival chain, one bin)."""
    rng = np.random.default_rng(seed)
    th = np.array(THETA_FULL) * (1 + rng.uniform(-0.05, 0.05, (64, 6)))
    s12, s13, d21, d32 = (th[:, k, None] for k in (0, 1, 4, 5))
    x, w = np.polynomial.legendre.leggauss(64)
    E = 0.5 * (e[0] + e[1]) + 0.5 * (e[1] - e[0]) * x
    w = w * np.exp(0.87 - 0.16 * E - 0.091 * E * E)
    om = oracle.baseline_weights(np.array(L))
    S = [sum(o * (w * np.sin(1266.932679419849 * d * Lr / E) ** 2).sum(axis=1) for o, Lr in zip(om, L))
         for d in (d21, d21 + d32, d32)]
    s12, c13, s13 = s12[:, 0], 1 - s13[:, 0], s13[:, 0]
    t = 4 * np.array([(1 - 2 * s12) * c13 ** 2 * S[0], -c13 * s13 * S[1], c13 * s13 * S[2]])
    return np.sqrt((np.abs(t).sum(axis=0) ** 2).mean() / (t.sum(axis=0) ** 2).mean())


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("n", [50, 262, 1000])
@pytest.mark.parametrize("nL", [1, 8])
def test_derivatives_are_contracted_in_pairs(api, nL, n, prec):
    """The derivative by s2_12 takes two pairs' sums with opposite signs: it is
    formed from float pairs, as the prediction.  Four FP32 roundings of the
    result (2^-25 each, rms: 6e-8; 9e-8 allowed), and of the terms the sums'
    own errors: below 1e-8 each (the terms in FP32 would add 2.5e-8)."""
    L = [23.2, 11.4, 44.9, 18.3, 45.1, 0.9, 22.2, 19.3][:nL]
    for lo, w in ((3.004, 0.4028), (7.265, 0.0145), (9.77, 0.4028)):
        e = np.array([lo, lo + w])
        mu, s12, s13, dm21, _ = derivative_errors(api, e, L, n, prec)
        k = s12_cancellation(e, L)
        assert mu < 5e-8 and s12 < 9e-8 + 1e-8 * k and s13 < 9e-8 and dm21 < 9e-8, (lo, k, mu, s12, s13, dm21)


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("n", [8, 100, 1000])
@pytest.mark.parametrize("channel", [("e", "tau", False), ("mu", "e", True)])
def test_cp_terms_cancel_exactly(api, channel, n, prec):
    """At short baselines the three CP terms sin y_21 + sin y_32 - sin y_31 of
    an appearance channel are fifteen times what is left of them: roundings of
    the single sums (2^-24 of each, 8e-8 of mu and more) must not remain.  What
    remains is that of T and of what pair 31 has beyond the others, 2^-25."""
    for lo, w in ((4167.0, 5.8), (3345.0, 5.8), (2426.0, 22.5)):
        mu = derivative_errors(api, np.array([lo, lo + w]), [810.0, 295.0], n, prec, channel, 1e-3)[0]
        assert mu < (3e-8 if n >= 100 else 6e-8), (lo, mu)  # few nodes: their own roundings do not average


@pytest.mark.parametrize("channel", [None, ("mu", "mu", False)])
def test_fit_layout_waits_for_the_first_fit(api, channel):
    """A plan that announces no data sets of its own holds 12 bytes per node
    until it is fitted (the mixed precisions' evaluations read no more), and its
    fits, captured into a graph too, equal those of a plan that announces them."""
    e, L, counts = np.linspace(1.8, 8.0, 33), [52.5], [40001, 40004]
    th = np.array([0.307, 0.0218, 7.53e-5, 2.44e-3] if channel is None else THETA_FULL)
    start = np.repeat(th[None] * 1.01, 2, 0)
    bytes_, res = {}, {}
    for m in (0, 2):
        plan = api.Plan(e, L, npts=2, node_counts=counts, prec="ff", kind="poisson", norm=1e4, max_datasets=m, channel=channel)
        f = plan.eval if channel is None else plan.eval_general
        data = f(plan.params_tensor(np.repeat(th[None], 2, 0)), dev(np.ones(32)), mu=True)["mu"].clone()
        bytes_[m] = plan.info()["device_bytes"]
        p, c = plan.params_tensor(start), torch.empty(2, dtype=torch.float64, device="cuda")
        if m:
            plan.fit(p, data, iters=3, chi2_out=c)
        else:
            p0 = p.clone()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                p.copy_(p0)
                plan.fit(p, data, iters=3, chi2_out=c, graph=False)
            graph.replay()
        res[m] = p.cpu().numpy(), c.cpu().numpy()
        assert plan.info()["device_bytes"] == bytes_[2] if m else plan.info()["device_bytes"] > bytes_[0]
        plan.status()
        plan.close()
    nodes = 32 * sum(counts)
    assert bytes_[0] < 12.1 * nodes + 4e6 and bytes_[2] - bytes_[0] == 16 * nodes
    for a, b in zip(res[0], res[2]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nbins,n", [(33, 65000), (64, 1031), (40, 50)])
def test_fp64_split_mapping_reads_either_layout(api, nbins, n):
    """A default GNA_FP64 plan keeps one copy of its nodes: its split mapping
    reads the bin mapping's layout, with the same results bit for bit as on a
    plan that has the split mapping's own."""
    e, L = np.linspace(1.8, 8.0, nbins + 1), [52.5, 30.0]
    th = np.repeat(np.array([[0.307, 0.0218, 7.53e-5, 2.44e-3]]), 2, 0)
    plans = {m: api.Plan(e, L, nodes_per_bin=n, npts=2, norm=1e4, prec="fp64", kind="poisson", max_datasets=2, mapping=m)
             for m in (None, "split")}
    assert plans[None].info()["device_bytes"] - plans["split"].info()["device_bytes"] < 16 * 31 * n + 40e6  # bins in groups, slices
    data = plans["split"].eval(plans["split"].params_tensor(th), dev(np.ones(nbins)), mu=True)["mu"].clone().round()
    plans[None].tuning = "mapping=split"
    out = {}
    for m, plan in plans.items():
        o = plan.eval(plan.params_tensor(th), data, grad=True, mu=True, spectra=True)
        p, c = plan.fit(plan.params_tensor(1.01 * th), data, iters=3)
        out[m] = [x.cpu().numpy() for x in (o["chi2"], o["grad"], o["mu"], o["spectra"], p, c)]
        plan.status()
        plan.close()
    for a, b in zip(out[None], out["split"]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["fp64", "f64phase", "ff"])
@pytest.mark.parametrize("zero", [0, 1])
@pytest.mark.parametrize("nL", [1, 3, 9])
def test_a_splitting_of_zero(api, nL, zero, prec):
    # one pair's phases, and their sums, vanish for every baseline: compensated
    # sums of zeros, chunks as long as they get (33 nodes: one and a rest)
    rng = np.random.default_rng(nL)
    e, n = np.linspace(3.0, 3.4, 38), 33
    L = rng.uniform(1.0, 60.0, nL)
    theta = np.array(wl.TRUTH)
    theta[2 + zero] = 0.0
    Nn = oracle.norm_for_total(e, n, L, wl.TRUTH)
    data = wl.poisson_data(Nn * (oracle.baseline_weights(L) @ oracle.binned(e, n, L, wl.TRUTH)), 7)
    ref = oracle.chain(e, n, L, theta, Nn, data, wl.POISSON)
    plan = api.Plan(e, L, nodes_per_bin=n, norm=Nn, prec=prec, kind="poisson")
    out = plan.eval(plan.params_tensor(theta), dev(data), grad=True, mu=True, spectra=True)
    plan.status()
    plan.close()
    assert rel(out["mu"][0].cpu().numpy(), ref["mu"]) < TOL[prec]
    assert rel(out["spectra"][0].cpu().numpy(), ref["mu_rb"]) < TOL[prec]
    assert normrel(out["grad"][0].cpu().numpy(), ref["grad"][:4]) < GTOL[prec]
    check_chi2(out["chi2"][0].item(), ref, data, wl.POISSON, TOL[prec], tag="zero splitting %d %d" % (nL, zero), plain=False)


@pytest.mark.parametrize("channel", [None, ("mu", "mu", False), ("mu", "e", True)])
@pytest.mark.parametrize("nL", [1, 3])
@pytest.mark.parametrize("L", [1e5, 2.2e6, 4.1e6, 7.3e6, 1e7])
@pytest.mark.parametrize("wide", [False, True])
def test_double_float_phases_far_out(api, L, nL, channel, wide):
    """Phases up to 2^22 pi (x about L at 3 MeV) in the double-float mode, on
    chunks of nodes and on nodes by themselves (wide): their error grows with
    the phase, q 5.1e-12 from the reduction (q half-turns) and 2^-46 of the
    phase from the product, and nothing else is added."""
    e = np.linspace(3.0, 3.0 + (3.0 if wide else 3e2) / L, 33)
    th = [0.307, 0.0218, 7.53e-5, 2.44e-3] if channel is None else THETA_FULL
    mu = {}
    for prec in ("fp64", "ff"):
        plan = api.Plan(e, L * (1 + 1e-3 * np.arange(nL)), nodes_per_bin=8 if wide else 64, prec=prec, kind="poisson", channel=channel)
        f = plan.eval if channel is None else plan.eval_general
        mu[prec] = f(plan.params_tensor(th), dev(np.ones(32)), mu=True)["mu"][0].cpu().numpy()
        plan.status()
        plan.close()
    x = 1266.932679419849 * 2.52e-3 * L * 1.002 / 3.0
    W = np.exp(0.87 - 0.48 - 0.819) * (e[1] - e[0])
    assert np.abs(mu["ff"] - mu["fp64"]).max() < W * (1e-7 + 2 * x * (5.2e-12 / np.pi + 2.0 ** -46))


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("general", [False, True])
def test_one_minus_cosine_keeps_its_relative_error(api, general, prec):
    """Near an oscillation minimum at maximal mixing the prediction is a sum of
    1 - cos r: the polynomial holds to 2.1e-8 of it (any channel; 4.2e-9 in the
    survival chain), which the mean over bins and points shows; what else there
    is, roundings of 6e-8 in each of 64 x 40 sums, averages to 2e-9."""
    K = 1e3 / (4 * 0.1973269804)
    L, dm = 52.5, 7.53e-5
    E0 = K * dm * L / (np.pi / 2)
    e = E0 / (1 + np.linspace(0.15, 0.03, 41) * 2 / np.pi)  # x = pi/2 + 0.03 .. 0.15
    th = np.array([[0.5, 1e-15, 0.5, 0.3, dm, 1e-12]] if general else [[0.5, 0.0, dm, 0.0]])
    th = np.repeat(th, 64, 0)
    th[:, 4 if general else 2] *= 1 + np.linspace(0.0, 1e-3, 64)
    mu = {}
    for p in ("fp64", prec):
        plan = api.Plan(e, [L], nodes_per_bin=33, npts=64, prec=p, kind="poisson", channel=("e", "e", False) if general else None)
        f = plan.eval_general if general else plan.eval
        mu[p] = f(plan.params_tensor(th), dev(np.ones(40)), mu=True)["mu"].cpu().numpy()
        plan.status()
        plan.close()
    mean = float((mu[prec] / mu["fp64"] - 1).mean())
    # the survival chain's double-float reduction rounds p - pi to 2^-29 (r below
    # 2^-3) with the same low bits at every point, those of pi's second part:
    # up to twice that over r = 0.06 .. 0.3
    same = 2 * 2.0 ** -29 / 0.1 if prec == "ff" and not general else 0.0
    assert abs(mean) < (2.1e-8 if general else 4.2e-9) + 6e-9 + same, mean


@pytest.mark.parametrize("prec", ["f64phase", "ff"])
@pytest.mark.parametrize("channel", [("mu", "mu", True), ("mu", "e", False)])
@pytest.mark.parametrize("n", [12, 30])
def test_one_chunk_between_quadrants(api, channel, n, prec):
    """Bins that are one chunk whose doubled phase 32 lies near 3 pi / 4, where
    sin r and cos r - 1 are largest: they are summed as differences from the
    anchor's values.  Left are the nodes' own roundings: three of 2^-25 / sqrt 3
    in a sine of 0.7, over P = 0.15 (nu_mu -> nu_mu) and averaged over n nodes:
    1.4e-7 / sqrt n, less where P is a small part of the sines (seen: half of it,
    0.8e-7 / sqrt n allowed for nu_mu -> nu_e).  Sums of the sines themselves
    gave 2.4e-7 / sqrt n and 1.8e-7 / sqrt n."""
    e = np.linspace(2150.0, 2300.0, 13)
    err = [derivative_errors(api, e[i:i + 2], [810.0], n, prec, channel, 1e-3, seed=i)[0] for i in range(12)]
    assert np.sqrt(np.mean(np.square(err))) < (1.4e-7 if channel[1] == "mu" else 0.8e-7) / np.sqrt(n), err
