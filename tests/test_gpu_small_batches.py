"""Binning of batches of small structures, a CTA per structure, at the sizes
where the choice between it and the kernels over all atoms lies, with empty and
one-atom structures, every kind of periodicity and structures many cells away
from their cell.  The same structures go through both by adding a large one."""
import numpy as np
import pytest

from paper_2303_12980_gb300 import synth
from tests.parity import FEAT_TOL, feature_errors

pytestmark = pytest.mark.gpu

PBC = [(1, 1, 1), (0, 0, 0), (1, 1, 0), (0, 1, 0)]


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


def _batch(sizes, seed):
    rng = np.random.default_rng(seed)
    pos, cells, pbc = [], [], []
    for s, n in enumerate(sizes):
        edge = (max(n, 4) / 0.08) ** (1 / 3)
        cell = np.eye(3) * edge * rng.uniform(0.8, 1.3, 3)
        if s % 3 == 2:
            cell = cell + rng.uniform(-0.2, 0.2, (3, 3)) * edge
        far = rng.integers(-40, 40, 3) * np.array(PBC[s % 4])
        pos.append((rng.uniform(0, 1, (n, 3)) + far) @ cell)
        cells.append(cell)
        pbc.append(PBC[s % 4])
    n = sum(sizes)
    return synth.Workload("small", np.concatenate(pos), np.stack(cells), np.array(pbc, np.uint8),
                          np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), rng.integers(0, 3, n).astype(np.int32),
                          *synth.gaussian_table(rng, [3, 4, 5], 2), [0, 1, 2], [0.4, 0.8], 4.5)


def _dev(torch, w):
    return torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc


@pytest.mark.parametrize("sizes", [[1], [7, 0, 1, 33, 64, 2, 255, 256], [128, 129, 31, 32, 127] * 40, [256, 257], [512] * 16,
                                   [512] * 15 + [511], [513] * 16], ids=lambda s: "%dx%d" % (len(s), max(s)))
def test_small_batches(torch, oracle_mod, sizes):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    w = _batch(sizes, 11)
    big = _batch(list(sizes) + [1500], 11)
    n = w.n_atoms
    # (the random draws of the two agree on the structures, not on the species)
    assert np.array_equal(big.positions[:n], w.positions)
    big.species[:n] = w.species
    F = GMPFeaturizer.from_workload(w)
    off, j, shift = (x.cpu().numpy() for x in F.neighbors(*_dev(torch, w)))
    boff, bj, bshift = (x.cpu().numpy() for x in F.neighbors(*_dev(torch, big)))
    assert np.array_equal(off, boff[: n + 1])
    assert np.array_equal(j, bj[: off[-1]]) and np.array_equal(shift, bshift[: off[-1]])
    centers = np.arange(0, n, max(1, n // 60))
    ref, fabs = oracle_mod.features(w, centers=centers, want_abs=True)
    for _ in range(2):  # lists counted first, then in one pass
        f = F.featurize(*_dev(torch, w)).cpu().numpy()[centers]
        assert feature_errors(f, ref, fabs).max() <= FEAT_TOL


@pytest.mark.parametrize("large", [False, True])
def test_points_of_empty_and_small_structures(torch, oracle_mod, large):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    w = _batch([0, 5, 0, 40] + ([700] if large else []), 3)
    rng = np.random.default_rng(5)
    S = len(w.cells)
    p_off = np.arange(S + 1, dtype=np.int64) * 6
    pts = np.concatenate([rng.uniform(-1, 2, (6, 3)) @ w.cells[s] for s in range(S)])
    ref, fabs = oracle_mod.point_features(w, pts, np.repeat(np.arange(S), 6), want_abs=True)
    f = GMPFeaturizer.from_workload(w).featurize_points(*_dev(torch, w), torch.from_numpy(pts).cuda(), p_off).cpu().numpy()
    assert (np.abs(f - ref) <= 1e-5 * np.maximum(np.maximum(np.abs(ref), 1e-6 * fabs), 2.0 ** -126)).all()
