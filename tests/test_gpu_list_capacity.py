"""Neighbor lists whose capacity, guessed from the handle's last batch, does not
fit the device: they are counted instead."""
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


@pytest.mark.parametrize("call", ["features", "vjp", "points"])
def test_guess_beyond_the_memory(torch, call):
    """10,000 atoms within one cutoff, then 1,000,000 centers with an atom each:
    as many pairs a center would take 360 GB."""
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(2)
    table = synth.gaussian_table(rng, [3], 2)
    n, m, rc = 10_000, 1_000_000, 5.0
    blob = rng.uniform(-1.4, 1.4, (n, 3))
    grid = np.stack(np.unravel_index(np.arange(m), (100, 100, 100)), 1) * 8.0
    one = torch.zeros(m, dtype=torch.int32, device="cuda")

    def run(F, pos):
        a = (torch.from_numpy(pos).cuda(), one[: len(pos)], [0, len(pos)], np.zeros((1, 3, 3)), [[0, 0, 0]])
        if call == "features":
            return F.featurize(*a)
        if call == "vjp":
            return torch.cat(F.featurize_vjp(*a, torch.ones((len(pos), F.num_features), device="cuda")), 1)
        pts = blob[:1] * 0.0 if pos is blob else grid[:, ::-1] + 0.25
        return F.featurize_points(*a, torch.from_numpy(np.ascontiguousarray(pts)).cuda(), [0, len(pts)])

    new = lambda: GMPFeaturizer([0], [0.5], rc, *table)
    F = new()
    run(F, blob)
    want = run(new(), grid)
    for _ in range(2):
        got = run(F, grid)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
