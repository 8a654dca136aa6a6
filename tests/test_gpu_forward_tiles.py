"""The forward kernel's tiles of 16 and 32 pairs sum the same terms in the same
order: features, and gradients from their moments, agree to the bit.  List
lengths around both tiles, one and several elements a list (pairs of a lane that
agree and that do not), coefficients of both signs, every shape.  (The density
of order -1 is summed by lanes, in another order.)"""
import numpy as np
import pytest

from paper_2303_12980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


@pytest.mark.parametrize("n_el", [1, 5])
@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("lmax,n_sig", [(0, 8), (1, 5), (2, 4), (2, 8), (3, 7), (4, 8), (2, 16), (3, 16), (4, 13), (5, 8), (6, 16)])
def test_tiles_agree(torch, lmax, n_sig, signed, n_el):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(100 * lmax + n_sig)
    sizes = [1, 2, 15, 16, 17, 18, 31, 32, 33, 34, 47, 48, 49, 64, 65, 97]  # every atom sees its whole cluster
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pos = rng.uniform(0, 2.8, (off[-1], 3))
    n_gauss, coef, expo = synth.gaussian_table(rng, [3, 4, 5, 6, 7][:n_el], 3)
    if signed:
        coef = coef * np.where(np.arange(len(coef)) % 3 == 1, -0.3, 1.0)
    S = len(sizes)
    w = synth.Workload("tiles", pos, np.zeros((S, 3, 3)), np.zeros((S, 3), np.uint8), off,
                       rng.integers(0, n_el, off[-1]).astype(np.int32), n_gauss, coef, expo, list(range(lmax + 1)),
                       [float(s) for s in np.geomspace(0.2, 1.2, n_sig)], 5.0)
    args = (torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc)
    g = torch.from_numpy(synth.upstream_gradient(w.n_atoms, w.n_features, seed=1)).cuda()
    F, got = GMPFeaturizer.from_workload(w), []
    for tile in (16, 32):
        vals = list(F.tuning())
        vals[0::6] = [tile] * (len(vals) // 6)
        F.set_tuning(vals)
        got.append([F.featurize(*args), *F.featurize_vjp(*args, g)])
    for a, b in zip(*got):
        assert torch.isfinite(a).all() and torch.equal(a, b)
