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


def test_outgrown_lists_are_not_computed_on(torch):
    """A batch with a fifth more pairs than the last one outgrows the guess: its
    forward kernels together take about as long as the one of a batch that fits."""
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(3)
    table = synth.gaussian_table(rng, [3, 5], 6)

    def batch(a):
        pos, cell = synth.fcc_supercell(rng, a, (20, 20, 20), 0.1)
        sp = torch.from_numpy(rng.integers(0, 2, len(pos)).astype(np.int32)).cuda()
        return torch.from_numpy(pos).cuda(), sp, [0, len(pos)], cell[None], [[1, 1, 1]]

    dense, sparse = batch(3.7), batch(3.95)
    F = GMPFeaturizer(list(range(7)), np.geomspace(0.05, 1.5, 16), 8.0, *table)
    want = F.featurize(*dense)

    def forward_ms(n):
        F.profile(True)
        got = F.featurize(*dense)
        torch.cuda.synchronize()
        ms, count = F.profile_read()["features"]
        F.profile(False)
        assert count == n and torch.equal(got, want)
        return ms

    fits = min(forward_ms(1) for _ in range(3))
    outgrown = []
    for _ in range(3):
        F.featurize(*sparse)
        outgrown.append(forward_ms(2))
    assert min(outgrown) < 1.4 * fits  # 1.9 when the partial lists are computed on


def test_query_of_the_rows(torch):
    """A Jacobian call whose buffers hold fewer rows than there are centers reads
    their number and computes no features."""
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(5)
    pos, cell = synth.fcc_supercell(rng, 3.6, (3, 3, 3), 0.1)
    n = len(pos)
    a = (torch.from_numpy(pos).cuda(), torch.zeros(n, dtype=torch.int32, device="cuda"), [0, n], cell[None], [[1, 1, 1]])
    F = GMPFeaturizer([0, 1, 2], [0.4, 0.8], 5.0, *synth.gaussian_table(rng, [3], 2))
    F.profile(True)
    first = F.featurize_grad(*a)  # asks for the rows, then takes them
    torch.cuda.synchronize()
    assert F.profile_read()["features"][1] == 1
    for b, e in ((0, n), (5, 9), (3, 3)):
        F._rows["grad"] = 0
        got = F.featurize_grad(*a, centers=(b, e))
        lo, hi = int(first[1][b]), int(first[1][e])
        assert torch.equal(got[0], first[0][b:e]) and torch.equal(got[1], first[1][b:e + 1] - lo)
        assert torch.equal(got[2], first[2][lo:hi]) and torch.equal(got[3], first[3][lo:hi])


@pytest.mark.parametrize("n_el", [1, 9000])
@pytest.mark.parametrize("rc", [12.8, 15.5, 15.9])  # 8,733, 15,515 and 16,831 images
def test_longest_list(torch, n_el, rc):
    """One atom in a cell of 1 A: lists of its images up to 16,384, the limit that the
    error names, whatever the number of elements."""
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    F = GMPFeaturizer([0], [0.5], rc, *synth.gaussian_table(np.random.default_rng(1), [3] * n_el, 1))
    a = (torch.zeros((1, 3), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"), [0, 1],
         np.eye(3)[None], [[1, 1, 1]])
    k = np.arange(-16, 17)
    x = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    x = x[(x * x).sum(1) < rc * rc]
    for _ in range(2):
        if len(x) > 16384:
            with pytest.raises(GMPError, match=f"{len(x)} neighbor images .limit 16384."):
                F.neighbors(*a)
            continue
        off, j, s = F.neighbors(*a)
        assert off.tolist() == [0, len(x)] and np.array_equal(s.cpu().numpy(), x) and not j.any()
        if n_el == 1:
            assert np.isfinite(F.featurize(*a).cpu().numpy()).all()
