"""The fit's device eigensolver (Section 3.1, "Linear transform": the PCA matrix comes from the
covariance of calibration data) against what the mathematics fixes -- numpy's symmetric solver,
orthonormality, the decomposition itself, a matrix built from a known spectrum -- against the
library's host solver, and the fit that uses it against the host-solver fit and the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1905_10830_b200 as tc
from synth import featuremaps as fm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


def _sym(n, seed, decay=0.9):
    """Q diag(lambda) Q^T with a geometric spectrum and a random orthogonal Q."""
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = 3.0 * decay ** np.arange(n)
    return (q * lam) @ q.T, lam, q


def _check_conventions(a, evals, evecs):
    n = a.shape[0]
    scale = max(1.0, np.abs(evals).max())
    assert np.all(np.diff(evals) <= 0.0)                                        # descending
    assert np.abs(evecs @ evecs.T - np.eye(n)).max() <= 1e-12                   # orthonormal rows
    assert np.abs(evecs @ a @ evecs.T - np.diag(evals)).max() <= 2e-13 * scale * max(1, n / 64)
    big = np.abs(evecs).argmax(axis=1)
    assert np.all(evecs[np.arange(n), big] > 0.0)                               # sign convention


@pytest.mark.parametrize("n", [1, 2, 3, 17, 64, 96, 255, 256, 511, 1024])
def test_device_eigh_against_numpy_and_the_host_solver(ctx, n):
    a, lam, _ = _sym(n, 900 + n)
    a = (a + a.T) / 2
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    assert 1 <= sweeps <= 60 or n == 1
    _check_conventions(a, evals, evecs)
    bound = 1e-13 * max(1, n / 16) * lam.max()           # absolute accuracy: a few hundred eps |A| at n = 1024
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= bound
    assert np.abs(evals - lam).max() <= bound                                   # the spectrum it was built from
    h_evals, h_evecs = tc.tc_host_eigh(a)
    assert np.abs(evals - h_evals).max() <= bound
    # eigenvectors of well separated eigenvalues agree with the host solver's (same sign rule)
    gap_ok = np.ones(n, dtype=bool)
    if n > 1:
        gaps = np.minimum(np.r_[np.inf, -np.diff(h_evals)], np.r_[-np.diff(h_evals), np.inf])
        gap_ok = gaps > 1e-4 * lam.max()
    assert np.abs(evecs[gap_ok] - h_evecs[gap_ok]).max() <= 1e-8


def test_device_eigh_rank_deficient_and_repeated(ctx):
    rng = np.random.default_rng(77)
    b = rng.standard_normal((40, 12))
    a = b @ b.T                                   # rank 12 of 40: 28 null directions
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    assert sweeps <= 20
    _check_conventions(a, evals, evecs)
    assert np.abs(evals[12:]).max() <= 1e-12 * evals[0]
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= 1e-12 * evals[0]
    # a multiple of the identity: nothing to rotate, one sweep, unit vectors
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.eye(9, dtype=torch.float64, device="cuda") * 2.5)
    assert sweeps == 1 and torch.all(evals == 2.5) and torch.equal(evecs, torch.eye(9, dtype=torch.float64, device="cuda"))
    # a diagonal matrix out of order: sorted, vectors are the unit vectors in that order
    d = torch.tensor([1.0, 5.0, 3.0], dtype=torch.float64, device="cuda")
    evals, evecs, _ = tc.tc_device_eigh(ctx, torch.diag(d))
    assert evals.tolist() == [5.0, 3.0, 1.0]
    assert torch.equal(evecs, torch.tensor([[0, 1, 0], [0, 0, 1], [1, 0, 0]], dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("dtype,basis_dtype,c", [(torch.float32, None, 64), (torch.bfloat16, None, 128),
                                                 (torch.bfloat16, tc.binding.TC_INT8, 64), (torch.bfloat16, None, 320)])
def test_fit_on_the_device_matches_the_host_solver_fit_and_the_oracle(ctx, dtype, basis_dtype, c):
    params = fm.layer_params(fm.LayerSpec(c, 8, 8, 0.92, None, 9100 + c))
    cal = fm.make_maps(params, 12, calib=True, dtype=dtype)
    dev = tc.tc_model_export(tc.tc_fit_pca(ctx, cal.cuda(), 5, basis_dtype=basis_dtype, eigensolver=tc.TC_EIG_DEVICE))
    host = tc.tc_model_export(tc.tc_fit_pca(ctx, cal.cuda(), 5, basis_dtype=basis_dtype, eigensolver=tc.TC_EIG_HOST))
    rounding = {None: "bf16" if dtype == torch.bfloat16 else "f32", tc.binding.TC_INT8: "int8"}[basis_dtype]
    want = oracle.fit_pca(cal, 5, basis_round=rounding, zero_level=True)
    assert np.array_equal(dev["mean"], host["mean"])
    for other in (host["basis"], want.basis):
        # the solvers agree to rounding: an entry may land on the neighbouring representable value
        # where its exact value sits at a rounding tie; directions of near-equal eigenvalues excepted
        gaps = np.minimum(np.r_[np.inf, -np.diff(want.eig)], np.r_[-np.diff(want.eig), np.inf])
        rows = gaps > 1e-9 * want.eig[0]
        mine, theirs = dev["basis"][rows], other[rows]
        if rounding == "int8":                     # compare the integers: the scales differ in their last bits
            mine = np.rint(mine / dev["basis_scale"])
            theirs = np.rint(theirs / (host["basis_scale"] if other is host["basis"] else want.basis_scale))
        ulp = {"bf16": 2.0 ** -8, "f32": 2.0 ** -23, "int8": 1.0}[rounding]
        assert np.abs(mine - theirs).max() <= ulp
        assert (mine == theirs).mean() >= 0.999
    assert np.allclose(dev["eig"], host["eig"], rtol=0, atol=1e-12 * host["eig"][0])
    assert np.isclose(dev["basis_scale"], host["basis_scale"], rtol=1e-12)
    assert np.isclose(dev["lo"], host["lo"], rtol=1e-9, atol=1e-12) and np.isclose(dev["step"], host["step"], rtol=1e-9)
    assert np.isclose(dev["lo"], want.lo, rtol=1e-6, atol=1e-6) and np.isclose(dev["step"], want.step, rtol=1e-6)


def test_online_fit_finishes_on_the_device(ctx):
    params = fm.layer_params(fm.LayerSpec(96, 6, 6, 0.9, None, 9300))
    cal = fm.make_maps(params, 20, calib=True, dtype=torch.bfloat16).cuda()
    st = tc.tc_fit_state_create(ctx, 96)
    for lo, hi in ((0, 7), (7, 20)):
        tc.tc_fit_state_update(ctx, st, cal[lo:hi])
    online = tc.tc_model_export(tc.tc_fit_state_finish(ctx, st, cal, 4))
    online_host = tc.tc_model_export(tc.tc_fit_state_finish(ctx, st, cal, 4, eigensolver=tc.TC_EIG_HOST))
    oneshot = tc.tc_model_export(tc.tc_fit_pca(ctx, cal, 4))
    for other in (online_host, oneshot):
        assert np.allclose(online["mean"], other["mean"], rtol=1e-12, atol=1e-12)
        assert np.allclose(online["eig"], other["eig"], rtol=0, atol=1e-10 * other["eig"][0])
        assert np.abs(online["basis"] - other["basis"]).max() <= 2.0 ** -8
        assert (online["basis"] == other["basis"]).mean() >= 0.999
        assert np.isclose(online["lo"], other["lo"], rtol=1e-6, atol=1e-6) and np.isclose(online["step"], other["step"], rtol=1e-6)


@pytest.fixture(params=[1])
def jacobi(ctx, request):
    tc.tc_force_jacobi(ctx, request.param)
    yield
    tc.tc_force_jacobi(ctx, 0)


@pytest.mark.parametrize("jacobi", [0, 1], indirect=True, ids=["division", "jacobi"])
@pytest.mark.parametrize("n", [2, 3, 5])
def test_rotations_are_orthogonal_to_fp64(ctx, jacobi, n):
    # Few columns, angles of every size: cosine and tangent of a rotation start from fp32 (1e-7), and a rotation that is
    # orthogonal to that only would leave 1e-7 |A| beside the diagonal.  Inner products stop at 8 sqrt(16) eps of the
    # norms, which (1.25 + 1) |A|_F turns into at most 2.25 times that; as much again for the rounding of the sweeps.
    rng = np.random.default_rng(70 + n)
    for i in range(60):
        a = rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-6, 0, (n, n))
        a = (a + a.T) / 2
        evals, evecs, _ = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
        evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
        bound = 4.5 * 8 * 4 * 2.0 ** -52
        assert np.abs(evecs @ evecs.T - np.eye(n)).max() <= bound
        assert np.abs(evecs @ a @ evecs.T - np.diag(evals)).max() <= bound * np.linalg.norm(a)


# The method of devices that cannot hold the clusters, at the first and the last size of each of its kernels.
@pytest.mark.parametrize("n", [1, 64, 65, 128, 129, 256, 257, 384, 385, 512, 513, 576])
def test_jacobi_at_the_edges_of_its_kernels(ctx, jacobi, n):
    a, lam, _ = _sym(n, 5000 + n, 0.97)
    a = (a + a.T) / 2
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    assert sweeps >= 1
    _check_conventions(a, evals, evecs)
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= 1e-13 * max(1, n / 16) * lam.max()


def test_fit_by_jacobi_matches_the_fit_by_division(ctx):
    params = fm.layer_params(fm.LayerSpec(96, 8, 8, 0.92, None, 9200))
    cal = fm.make_maps(params, 12, calib=True, dtype=torch.float32).cuda()
    default = tc.tc_model_export(tc.tc_fit_pca(ctx, cal, 5))
    tc.tc_force_jacobi(ctx, 1)
    other = tc.tc_model_export(tc.tc_fit_pca(ctx, cal, 5))
    tc.tc_force_jacobi(ctx, 0)
    assert np.array_equal(default["mean"], other["mean"])
    assert np.allclose(default["eig"], other["eig"], rtol=0, atol=1e-12 * default["eig"][0])
    assert np.abs(default["basis"] - other["basis"]).max() <= 2.0 ** -23 and (default["basis"] == other["basis"]).mean() >= 0.99


# Edges of the cluster solver: lanes' elements and blocks of the cluster change at multiples of 64, groups of
# eigenvectors at multiples of 16, halves of the division at powers of two; 576 rows are the last that fit, 577 take Jacobi.
@pytest.mark.parametrize("n", [4, 5, 15, 16, 31, 32, 33, 63, 65, 127, 129, 191, 193, 257, 300, 384, 385, 320, 321, 512, 513, 575, 576, 577])
def test_device_eigh_at_the_edges_of_its_kernels(ctx, n):
    a, lam, _ = _sym(n, 4000 + n, 0.97)
    a = (a + a.T) / 2
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    assert 1 <= sweeps <= 60
    _check_conventions(a, evals, evecs)
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= 1e-13 * max(1, n / 16) * lam.max()


def _rotated(lam, seed):
    q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((len(lam), len(lam))))
    return (q * lam) @ q.T


def _clustered(n):
    return _rotated(np.r_[np.ones(n // 2), 2 * np.ones(n // 3), np.arange(n - n // 2 - n // 3)], n)


# Eigenvalues that agree but for rounding, most of them at or beside a power of two: spreading them apart has to leave no two equal.
@pytest.mark.parametrize("n", [33, 64, 100, 150, 256, 384, 576])
@pytest.mark.parametrize("values", [(1.0, 2.0), (2.0, 1.0, 0.0), (-1.0, 1.0), (1.0,), (3.0, 0.0), (1.0 - 2.0 ** -53, 0.25, 2.0 ** -20), (-2.0, -1.0)],
                         ids=["1 2", "2 1 0", "-1 1", "1", "3 0", "below 1", "-2 -1"])
def test_device_eigh_of_a_few_values(ctx, n, values):
    a = _rotated(np.resize(np.array(values), n), n + len(values))
    a = (a + a.T) / 2
    evals, evecs, _ = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    norm = max(abs(v) for v in values)                  # bounds as in the next test
    assert np.abs(evecs @ evecs.T - np.eye(n)).max() <= 2 * n * 2.0 ** -52
    assert np.abs(evecs @ a @ evecs.T - np.diag(evals)).max() <= 4 * n * 2.0 ** -52 * norm
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= 4 * n * 2.0 ** -52 * norm


@pytest.mark.parametrize("a", [
    np.ones((64, 64)),                                                                     # rank 1
    np.diag(np.abs(np.arange(129) - 64.0)) + np.eye(129, k=1) + np.eye(129, k=-1),         # pairs that agree to rounding
    2 * np.eye(200) - np.eye(200, k=1) - np.eye(200, k=-1),                                # equal halves at every cut
    np.eye(100) + 1e-15 * (np.eye(100, k=1) + np.eye(100, k=-1)),                          # couplings at the rounding of the diagonal
    np.diag(np.r_[np.zeros(70), np.arange(1.0, 31.0)]),                                    # diagonal, most of it zero
    np.kron(np.eye(8), np.full((16, 16), 0.5)),                                            # uncoupled blocks
    _clustered(150), np.zeros((40, 40)), 1e-200 * _clustered(70), 1e200 * _clustered(70),
], ids=["ones", "wilkinson", "second difference", "tiny coupling", "diagonal", "blocks", "clusters", "zero", "small", "large"])
def test_device_eigh_of_repeated_and_uncoupled_eigenvalues(ctx, a):
    # Nothing is deflated: equal eigenvalues are set apart by one unit in the last place of |T| each, n of them by n / 2 eps |A| at
    # a level, twice that over all levels (n, n / 2, ...); products and the reduction add a few sqrt(n) eps, n for good measure.
    n = a.shape[0]
    a = (a + a.T) / 2
    evals, evecs, _ = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    norm = np.abs(np.linalg.eigvalsh(a)).max()
    assert np.all(np.diff(evals) <= 0.0)
    assert np.abs(evecs @ evecs.T - np.eye(n)).max() <= 2 * n * 2.0 ** -52
    assert np.abs(evecs @ a @ evecs.T - np.diag(evals)).max() <= 4 * n * 2.0 ** -52 * norm
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= 4 * n * 2.0 ** -52 * norm


@pytest.mark.parametrize("n", [3, 100, 700])
def test_device_eigh_refuses_what_is_not_finite(ctx, n):
    for bad in (float("nan"), float("inf")):
        a = torch.eye(n, dtype=torch.float64, device="cuda")
        a[n - 1, n - 2] = a[n - 2, n - 1] = bad
        with pytest.raises(tc.TcError):
            tc.tc_device_eigh(ctx, a)
