"""Atoms of one periodic structure more than 511 cells apart, each within 500 of
the first: the image index between them does not fit.  Every call reports it,
with lists counted first and in one pass, sorted and by species, and in a replayed graph,
and the handle stays usable."""
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


@pytest.mark.parametrize("on_dev", [True, False])
@pytest.mark.parametrize("axis,cells", [(0, (0, 400, -200)), (1, (0, 400, -200)), (2, (0, -400, 200)), (0, (0, 300, -220)),
                                        (2, (0, 300, -200))])
def test_image_beyond_the_packed_index(torch, axis, cells, on_dev):
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    rng = np.random.default_rng(8)
    pos = rng.uniform(0, 5.0, (3, 3))
    w = synth._single("far", pos, np.eye(3) * 5.0, [1, 1, 1], np.array([0, 1, 0], np.int32),
                      synth.gaussian_table(rng, [3, 4], 2), [0, 1, 2], [0.4, 0.8], 4.4)
    far = pos.copy()
    far[:, axis] += 5.0 * np.array(cells)
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()) if on_dev else np.ascontiguousarray
    fits = max(cells) - min(cells) <= 509  # (neighbors lie within two cells of one another)
    g = synth.upstream_gradient(3, w.n_features, seed=1)
    off = [0, 2]

    def calls(F, x):
        a = (put(x), put(w.species), w.atom_off, w.cells, w.pbc)
        return [lambda: F.featurize(*a), lambda: F.featurize_vjp(*a, put(g))[1], lambda: F.featurize_vjp_virial(*a, put(g))[2],
                lambda: F.featurize_grad(*a)[3], lambda: F.featurize_grad(*a, centers=(1, 3))[3], lambda: F.neighbors(*a)[1],
                lambda: F.featurize_points(*a, put(x[1:] + 0.1), off)]

    for k in range(7):
        F = GMPFeaturizer.from_workload(w)
        want = [torch.as_tensor(calls(F, pos)[q]()).cpu() for q in (0, k)]
        for _ in range(2):
            if fits:
                calls(F, far)[k]()
            else:
                with pytest.raises(GMPError, match="image index"):
                    calls(F, far)[k]()
        assert torch.equal(torch.as_tensor(calls(F, pos)[k]()).cpu(), want[1])
        assert torch.equal(torch.as_tensor(calls(F, pos)[0]()).cpu(), want[0])


def test_replayed_graph(torch):
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    rng = np.random.default_rng(8)
    pos = rng.uniform(0, 5.0, (3, 3))
    w = synth._single("far", pos, np.eye(3) * 5.0, [1, 1, 1], np.array([0, 1, 0], np.int32),
                      synth.gaussian_table(rng, [3, 4], 2), [0, 1, 2], [0.4, 0.8], 4.4)
    F, st = GMPFeaturizer.from_workload(w), torch.cuda.Stream()
    F.set_graph(True)
    buf, sp = torch.from_numpy(pos).cuda(), torch.from_numpy(w.species).cuda()
    out = torch.empty((3, w.n_features), device="cuda")
    torch.cuda.synchronize()
    run = lambda: F.featurize(buf, sp, w.atom_off, w.cells, w.pbc, out=out, stream=st)
    for _ in range(3):
        run()
    torch.cuda.synchronize()
    want = out.clone()
    buf += torch.tensor([[0.0, 0, 0], [2000.0, 0, 0], [-1000.0, 0, 0]], device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    with pytest.raises(GMPError, match="image index"):
        run()
    buf.copy_(torch.from_numpy(pos))
    torch.cuda.synchronize()
    run()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
