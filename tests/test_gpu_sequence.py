"""The launch sequence of a call: neighbor lists built with capacities guessed
from the handle's last build (batches that outgrow them, device and host
buffers, every kind of call), errors found by the deferred check, batch
descriptions that change from call to call, and the scan of the bin counts on
either side of its one-CTA limit."""
import numpy as np
import pytest

from paper_2303_12980_gb300 import synth
from tests.parity import FEAT_TOL, feature_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


def _wl(n_dense, seed=3, orders=(0, 1, 2), n_sig=3):
    """A sparse cluster (one pair of atoms) or a dense periodic crystal."""
    rng = np.random.default_rng(seed)
    table = synth.gaussian_table(rng, [4, 6], 3)
    sig = np.geomspace(0.2, 1.0, n_sig)
    if n_dense == 0:
        return synth._single("pair", np.array([[0., 0, 0], [1.5, 0, 0]]), np.zeros((3, 3)), [0, 0, 0],
                             np.array([0, 1], np.int32), table, orders, sig, 6.0)
    pos, cell = synth.fcc_supercell(rng, 3.6, (n_dense,) * 3, 0.1)
    return synth._single("fcc", pos, cell, [1, 1, 1], rng.integers(0, 2, len(pos)).astype(np.int32), table, orders, sig, 6.0)


def _calls(torch, F, w, on_dev):
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()) if on_dev else (lambda a: a)
    args = (put(w.positions), put(w.species), w.atom_off, w.cells, w.pbc)
    g = synth.upstream_gradient(w.n_atoms, w.n_features, seed=1)
    pts = w.positions[:5] + 0.3
    yield "features", lambda: [F.featurize(*args)]
    yield "vjp", lambda: list(F.featurize_vjp(*args, put(g)))
    yield "virial", lambda: list(F.featurize_vjp_virial(*args, put(g)))
    yield "points", lambda: [F.featurize_points(*args, put(pts), [0, len(pts)])]
    yield "jacobian", lambda: list(F.featurize_grad(*args))


@pytest.mark.parametrize("on_dev", [True, False])
@pytest.mark.parametrize("n_sig", [3, 18])
def test_lists_outgrow_the_guess(torch, on_dev, n_sig):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    sparse, dense = _wl(0, n_sig=n_sig), _wl(4, n_sig=n_sig)
    for (name, _), k in zip(_calls(torch, None, sparse, on_dev), range(5)):
        F, fresh = GMPFeaturizer.from_workload(sparse), GMPFeaturizer.from_workload(dense)
        first = [c for _, c in _calls(torch, F, sparse, on_dev)][k]
        first()
        again = [c for _, c in _calls(torch, F, dense, on_dev)][k]
        want = [c for _, c in _calls(torch, fresh, dense, on_dev)][k]()
        for got in (again(), again()):  # outgrown and counted; then within the new guess
            torch.cuda.synchronize()
            for a, b in zip(got, want):
                assert torch.equal(torch.as_tensor(a).cpu(), torch.as_tensor(b).cpu()), name


def test_error_found_after_launching(torch):
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    w = _wl(4)
    F = GMPFeaturizer.from_workload(w)
    pos, sp = torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda()
    ok = [F.featurize(pos, sp, w.atom_off, w.cells, w.pbc) for _ in range(2)]
    bad = sp.clone()
    bad[7] = 9
    with pytest.raises(GMPError, match="species"):
        F.featurize(pos, bad, w.atom_off, w.cells, w.pbc)
    nan = pos.clone()
    nan[3, 1] = float("nan")
    with pytest.raises(GMPError, match="non-finite"):
        F.featurize(nan, sp, w.atom_off, w.cells, w.pbc)
    with pytest.raises(GMPError):  # a description that is refused half-way
        F.featurize(pos, sp, w.atom_off, np.zeros((1, 3, 3)), w.pbc)
    assert torch.equal(F.featurize(pos, sp, w.atom_off, w.cells, w.pbc), ok[0]) and torch.equal(ok[0], ok[1])


@pytest.mark.parametrize("n", [8187, 8188, 8189])  # 2 n + 8 bins: 16382, 16384, 16386
@pytest.mark.parametrize("periodic", [True, False])
def test_bins_around_the_scan_limit(torch, oracle_mod, n, periodic):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(n)
    pos, cell = synth.fcc_supercell(rng, 3.6, (13, 13, 13), 0.1)
    pos = pos[rng.permutation(len(pos))[:n]]
    w = synth._single("scan", pos, cell, [int(periodic)] * 3, np.zeros(n, np.int32), synth.gaussian_table(rng, [4], 2),
                      [0, 1], [0.4, 0.8], 4.5)
    centers = np.arange(0, n, 211)
    ref, fabs = oracle_mod.features(w, centers=centers, want_abs=True)
    F = GMPFeaturizer.from_workload(w)
    f = F.featurize(torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc)
    assert feature_errors(f.cpu().numpy()[centers], ref, fabs).max() <= FEAT_TOL


@pytest.mark.parametrize("on_dev", [True, False])
@pytest.mark.parametrize("n_sig", [3, 18])  # 18: two passes over the same bins
@pytest.mark.parametrize("virial", [False, True])
def test_gradient_bins_are_left_empty(torch, on_dev, n_sig, virial):
    """Gradients of a handle whose bins held another batch, a refused call's
    sums, infinities, or grew in between, to the bit of a fresh handle's."""
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    small, large = _wl(2, n_sig=n_sig), _wl(4, n_sig=n_sig)
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()) if on_dev else (lambda a: a)

    def call(F, w, bad=False, scale=1.0):
        sp = w.species.copy()
        if bad:
            sp[-1] = 9
        g = (synth.upstream_gradient(w.n_atoms, w.n_features, seed=1) * np.float32(scale)).astype(np.float32)
        f = F.featurize_vjp_virial if virial else F.featurize_vjp
        return [torch.as_tensor(x).cpu() for x in f(put(w.positions), put(sp), w.atom_off, w.cells, w.pbc, put(g))]

    want = {id(w): call(GMPFeaturizer.from_workload(w), w) for w in (small, large)}
    F = GMPFeaturizer.from_workload(small)
    steps = [(small, {}), (small, {"scale": np.inf}), (small, {}), (small, {"bad": True}), (small, {}), (large, {}),
             (large, {"bad": True}), (small, {}), (large, {})]
    for w, how in steps:
        if how.get("bad"):
            with pytest.raises(GMPError, match="species"):
                call(F, w, **how)
            continue
        got = call(F, w, **how)
        if not how:
            for a, b in zip(got, want[id(w)]):
                assert torch.equal(a, b)
