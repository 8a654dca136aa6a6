"""Dense Jacobian rows of the kernel for orders up to 4 and of the general one
(5, 6) on a cell small enough that most rows sum several images: every highest
order, order subsets, the density, and sigma counts that fill a group of lanes,
leave some idle or need a second pass."""
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


@pytest.mark.parametrize("orders,n_sig", [([0], 1), ([1], 4), ([-1, 2], 5), ([3, 1], 8), ([0, 1, 2, 3, 4], 8), ([4], 16),
                                          ([4, -1, 0], 18), ([5, 2], 3), ([6], 9)])
def test_rows(torch, oracle_mod, orders, n_sig):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(10 * n_sig + orders[0])
    pos = synth.random_periodic_box(rng, 11, 5.1, 1.2)
    w = synth._single("cell", pos, np.diag([5.1, 5.1, 5.1]) + np.array([[0, 0.7, 0], [0, 0, 0], [-0.4, 0, 0]]), [1, 1, 1],
                      rng.integers(0, 3, 11).astype(np.int32), synth.gaussian_table(rng, [3, 5, 6], 3), orders,
                      np.geomspace(0.15, 1.1, n_sig) if n_sig > 1 else [0.5], 4.6)
    F = GMPFeaturizer.from_workload(w)
    args = (torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc)
    ref, fabs = oracle_mod.features(w, want_abs=True)
    off, j, jac, jabs = oracle_mod.jacobian_rows(w, want_abs=True)
    for _ in range(2):  # counted, then single-pass lists
        f, goff, gj, gjac = (x.cpu().numpy() for x in F.featurize_grad(*args))
        assert feature_errors(f, ref, fabs).max() <= FEAT_TOL
        assert np.array_equal(goff, off) and np.array_equal(gj, j)
        assert grad_errors(gjac, jac, jabs, tau=JAC_TAU).max() <= GRAD_TOL
