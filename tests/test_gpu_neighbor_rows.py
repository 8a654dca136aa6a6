"""Neighbor search over rows of bins: cells whose axes are orthogonal, along
the coordinate axes or rotated, and skew ones; boxes much smaller and larger
than the cutoff; a row that wraps along axis 0; more than 32 rows; clusters
and points beyond their atoms.  Sets bit for bit against the oracle."""
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


def _rotation(rng):
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    return q


def _cell(kind, rng, edge):
    c = np.diag(np.asarray(edge, np.float64))
    if kind == "rotated":
        c = c @ _rotation(rng)
    elif kind == "skew":
        c = c + np.array([[0, .6, -.4], [.3, 0, .5], [-.7, .2, 0]]) * min(edge)
    return c


@pytest.mark.parametrize("kind", ["axes", "rotated", "skew"])
@pytest.mark.parametrize("edge,n,pbc", [((3.1, 3.3, 2.9), 3, (1, 1, 1)), ((9.0, 30.0, 13.0), 150, (1, 1, 1)),
                                        ((41.0, 12.0, 8.0), 260, (1, 1, 0)), ((11.0, 11.0, 11.0), 60, (0, 1, 1)),
                                        ((16.0, 14.0, 15.0), 1500, (1, 1, 1))])
def test_neighbor_rows(torch, oracle_mod, kind, edge, n, pbc):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(n)
    cell = _cell(kind, rng, edge)
    pos = rng.uniform(-0.3, 1.3, (n, 3)) @ cell
    w = synth._single("rows", pos, cell, pbc, rng.integers(0, 3, n).astype(np.int32), synth.gaussian_table(rng, [3, 4, 5], 2),
                      [0], [0.6], 5.3)
    centers = np.arange(0, n, max(1, n // 40))
    off, j, shift = oracle_mod.neighbors(w, centers=centers)[:3]
    F = GMPFeaturizer.from_workload(w)
    dev = torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda()
    goff, gj, gs = (x.cpu().numpy() for x in F.neighbors(*dev, w.atom_off, w.cells, w.pbc))
    for k, i in enumerate(centers):
        a = np.concatenate([gj[goff[i]:goff[i + 1], None], gs[goff[i]:goff[i + 1]]], 1)
        b = np.concatenate([np.asarray(j[off[k]:off[k + 1]])[:, None], np.asarray(shift[off[k]:off[k + 1]]).reshape(-1, 3)], 1)
        assert np.array_equal(a[np.lexsort(a.T[::-1])], b[np.lexsort(b.T[::-1])])
    # the records grouped by species (features) against the sorted ones (Jacobian call), and
    # points away from the atoms
    ref, fabs = oracle_mod.features(w, centers=centers, want_abs=True)
    f = F.featurize(*dev, w.atom_off, w.cells, w.pbc).cpu().numpy()[centers]
    assert (np.abs(f - ref) <= 1e-5 * np.maximum(np.abs(ref), 1e-6 * fabs)).all()
    pts = rng.uniform(-1.5, 2.5, (40, 3)) @ cell
    pref, pabs = oracle_mod.point_features(w, pts, np.zeros(40, np.int64), want_abs=True)
    fp = F.featurize_points(*dev, w.atom_off, w.cells, w.pbc, torch.from_numpy(pts).cuda(), [0, 40]).cpu().numpy()
    assert (np.abs(fp - pref) <= 1e-5 * np.maximum(np.maximum(np.abs(pref), 1e-6 * pabs), 2.0 ** -126)).all()


@pytest.mark.parametrize("n", [1, 2, 3, 17, 32, 33, 34, 64, 65, 66, 129, 130, 257, 258, 600])
def test_sorted_lists(torch, oracle_mod, n):
    """n atoms all within the cutoff of one another (lists of n, the center's
    own entry included), and the same periodic along one axis (3 n): ascending
    (atom, image)."""
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(n)
    pos = rng.permutation(n)[:, None] * np.array([[0.002, 0.0, 0.0]]) + rng.uniform(0, 1e-3, (n, 3))
    for pbc in ([0, 0, 0], [0, 0, 1]):
        w = synth._single("line", pos, np.eye(3) * 3.7, pbc, np.zeros(n, np.int32), synth.gaussian_table(rng, [4], 2), [0],
                          [0.6], 4.0)
        F = GMPFeaturizer.from_workload(w)
        off, j, s = (x.cpu().numpy().astype(np.int64) for x in F.neighbors(
            torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc))
        s = s.reshape(-1, 3)
        key = ((j * 1024 + s[:, 0] + 512) * 1024 + s[:, 1] + 512) * 1024 + s[:, 2] + 512
        assert np.array_equal(off, oracle_mod.neighbors(w)[0]) and off[-1] == n * n * (3 if pbc[2] else 1)
        for i in range(0, n, max(1, n // 9)):
            assert (np.diff(key[off[i]:off[i + 1]]) > 0).all()
