"""The double-float refinement order by order: near-symmetric crystals, whose
features of one order cancel at every center, with sigma counts that leave the
last pair of sigmas of a queue entry half empty (1, 3) or start a second pass
(17)."""
import numpy as np
import pytest

from paper_2303_12980_gb300 import synth
from tests.parity import FEAT_TOL, GRAD_TOL, feature_errors, grad_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


@pytest.mark.parametrize("order,n_sig", [(1, 1), (2, 3), (3, 17), (4, 1), (4, 3), (5, 3), (6, 1), (6, 3)])
def test_refined_order(torch, oracle_mod, order, n_sig):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(40 + order)
    pos, cell = synth.fcc_supercell(rng, 3.9, (3, 3, 3), 1e-3)
    w = synth._single("fcc108", pos, cell, [1, 1, 1], np.zeros(len(pos), np.int32),
                      synth.gaussian_table(rng, [5], 6), [order], np.geomspace(0.2, 1.5, n_sig) if n_sig > 1 else [1.2], 7.5)
    ref, fabs = oracle_mod.features(w, want_abs=True)
    F = GMPFeaturizer.from_workload(w)
    dev = torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda()
    args = (*dev, w.atom_off, w.cells, w.pbc)
    f = F.featurize(*args)
    assert feature_errors(f.cpu().numpy(), ref, fabs).max() <= FEAT_TOL
    # the moments that the backward kernel reads are the refined ones
    g = synth.upstream_gradient(w.n_atoms, w.n_features, seed=order)
    f2, gp = F.featurize_vjp(*args, torch.from_numpy(g).cuda())
    assert torch.equal(f, f2)
    atoms = np.arange(0, w.n_atoms, 9)
    gref, gabs = oracle_mod.vjp_atoms(w, g, atoms, want_abs=True)
    assert grad_errors(gp.cpu().numpy()[atoms], gref, gabs).max() <= GRAD_TOL
