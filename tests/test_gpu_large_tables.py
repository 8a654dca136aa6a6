"""Element tables that leave room for few warps beside them in shared memory, or
for none of the kernels that stage the most a warp: the same results from those
that stage less, features and Jacobian rows against the oracle."""
import numpy as np
import pytest

from paper_2303_12980_gb300 import synth
from tests.parity import FEAT_TOL, GRAD_TOL, JAC_TAU, feature_errors, grad_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


def _workload(lmax, n_sig, n_el, n_gauss):
    rng = np.random.default_rng(n_el)
    n = 40
    pos = rng.uniform(0, 6.0, (n, 3))
    return synth._single("tables", pos, np.eye(3) * 6.0, [1, 1, 0], rng.permutation(np.arange(n) * (n_el - 1) // (n - 1)).astype(np.int32),
                         synth.gaussian_table(rng, rng.integers(1, 9, n_el), n_gauss), list(range(lmax + 1)),
                         np.geomspace(0.15, 1.0, n_sig), 3.5)


# the last table that one warp of a kernel fits beside, and the next; the largest
# that the smallest kernels do
@pytest.mark.parametrize("lmax,n_sig,n_el,n_gauss", [(2, 16, 52, 10), (2, 16, 53, 10), (2, 16, 66, 8), (2, 8, 99, 10), (3, 8, 87, 10),
                                                     (3, 8, 108, 8), (4, 16, 38, 10), (4, 16, 39, 10), (4, 16, 40, 10),
                                                     (4, 16, 33, 12), (4, 8, 96, 8), (1, 16, 63, 10), (0, 4, 290, 8)])
def test_large_tables(torch, oracle_mod, lmax, n_sig, n_el, n_gauss):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    w = _workload(lmax, n_sig, n_el, n_gauss)
    F = GMPFeaturizer.from_workload(w)
    a = (torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc)
    ref, fabs = oracle_mod.features(w, want_abs=True)
    f = F.featurize(*a).cpu().numpy()
    assert feature_errors(f, ref, fabs).max() <= FEAT_TOL
    g = synth.upstream_gradient(w.n_atoms, w.n_features, seed=1)
    atoms = np.arange(0, w.n_atoms, 3)
    gref, gabs = oracle_mod.vjp_atoms(w, g, atoms, want_abs=True)
    _, gp = F.featurize_vjp(*a, torch.from_numpy(g).cuda())
    assert grad_errors(gp.cpu().numpy()[atoms], gref, gabs).max() <= GRAD_TOL
    off, j, jac, jabs = oracle_mod.jacobian_rows(w, want_abs=True)
    _, goff, gj, gjac = (x.cpu().numpy() for x in F.featurize_grad(*a))
    assert np.array_equal(goff, off) and np.array_equal(gj, j)
    assert grad_errors(gjac, jac, jabs, tau=JAC_TAU).max() <= GRAD_TOL


# either side of the lines where the Jacobian kernel for orders up to 4 gives way
@pytest.mark.parametrize("lmax,n_sig,n_el,n_gauss", [(4, 16, 21, 10), (4, 16, 22, 10), (2, 4, 6, 4), (2, 4, 7, 4), (2, 16, 38, 10),
                                                     (2, 16, 39, 10)])
def test_rows_either_side(torch, oracle_mod, lmax, n_sig, n_el, n_gauss):
    test_large_tables(torch, oracle_mod, lmax, n_sig, n_el, n_gauss)


# the untuned forward tile of 32 pairs pays beside small tables only
@pytest.mark.parametrize("lmax,n_sig,n_el,n_gauss,tile", [(2, 8, 10, 8, 32), (2, 8, 40, 8, 16), (3, 7, 20, 4, 32), (3, 7, 6, 32, 16),
                                                          (4, 8, 3, 5, 32), (4, 8, 3, 16, 16), (4, 8, 10, 1, 16), (2, 16, 10, 4, 32),
                                                          (2, 16, 20, 4, 16), (1, 8, 1, 4, 16), (6, 16, 1, 4, 16)])
def test_untuned_tile(torch, lmax, n_sig, n_el, n_gauss, tile):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    F = GMPFeaturizer.from_workload(_workload(lmax, n_sig, n_el, n_gauss))
    assert F.tuning()[0] == tile
