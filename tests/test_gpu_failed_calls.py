"""A call that fails after its neighbor lists were queued (here: tables that no
compute kernel fits beside) leaves nothing of them to the next one."""
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


@pytest.mark.parametrize("call", ["features", "vjp", "jacobian", "points"])
@pytest.mark.parametrize("what", ["outgrown", "species"])
def test_no_condition_is_left(torch, call, what):
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    rng = np.random.default_rng(4)
    n_el = 2000
    table = synth.gaussian_table(rng, [3] * n_el, 1)
    pos, cell = synth.fcc_supercell(rng, 3.6, (4, 4, 4), 0.1)
    n = len(pos)
    put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sp = np.arange(n, dtype=np.int32)
    lone = (put(np.arange(2)[:, None] * np.array([[3.0, 0, 0]])), put(sp[:2]), [0, 2], np.zeros((1, 3, 3)), [[0, 0, 0]])
    dense = (put(pos), put(sp), [0, n], cell[None], [[1, 1, 1]])
    bad = (dense[0], put(sp + n_el - 5), *dense[2:])
    new = lambda: GMPFeaturizer([0], [0.5], 6.0, *table)
    want = new().neighbors(*dense)
    F = new()
    F.neighbors(*(lone if what == "outgrown" else dense))  # the capacities of the next lists
    a = dense if what == "outgrown" else bad
    calls = {"features": lambda: F.featurize(*a), "vjp": lambda: F.featurize_vjp(*a, torch.ones((n, 1), device="cuda")),
             "jacobian": lambda: F.featurize_grad(*a), "points": lambda: F.featurize_points(*a, a[0], [0, n])}
    with pytest.raises(GMPError):
        calls[call]()
    F.sync()
    for x, y in zip(F.neighbors(*dense), want):
        assert torch.equal(x, y)


@pytest.mark.parametrize("n", [2, 8])  # 32 and 2,048 atoms: one CTA a structure, or several kernels
def test_description_uploaded_on_another_stream(torch, n):
    """A call without points uploads the batch description behind what its stream
    holds, and returns; the next call, on another stream, waits for it."""
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(6)
    pos, cell = synth.fcc_supercell(rng, 3.6, (n, n, n), 0.1)
    w = synth._single("fcc", pos, cell, [1, 1, 0], rng.integers(0, 2, len(pos)).astype(np.int32),
                      synth.gaussian_table(rng, [3, 4], 2), [0, 1, 2], [0.4, 0.8], 5.0)
    a = (torch.from_numpy(w.positions).cuda(), torch.from_numpy(w.species).cuda(), w.atom_off, w.cells, w.pbc)
    want = GMPFeaturizer.from_workload(w).featurize(*a)
    F, s1, s2 = GMPFeaturizer.from_workload(w), torch.cuda.Stream(), torch.cuda.Stream()
    none = torch.empty((0, 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
    F.featurize_points(*a, none, [0, 0], stream=s1)
    got = F.featurize(*a, stream=s2)
    assert s1.query()
    s2.synchronize()
    assert torch.equal(got, want)


def test_nothing_is_in_flight_after_a_failure(torch):
    """A failed call returns when what it queued is done; a handle is destroyed only
    when its last upload is."""
    from paper_2303_12980_gb300.binding import GMPError, GMPFeaturizer
    rng = np.random.default_rng(4)
    pos, cell = synth.fcc_supercell(rng, 3.6, (3, 3, 3), 0.1)
    n = len(pos)
    a = (torch.from_numpy(pos).cuda(), torch.zeros(n, dtype=torch.int32, device="cuda"), [0, n], cell[None], [[1, 1, 1]])
    F = GMPFeaturizer([0, 1], [0.4], 5.0, *synth.gaussian_table(rng, [3], 2))
    F.featurize(*a)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)
    with pytest.raises(GMPError, match="species"):
        F.featurize(a[0], a[1] + 7, *a[2:], stream=s)
    assert s.query()
    none = torch.empty((0, 3), dtype=torch.float64, device="cuda")
    G = GMPFeaturizer([0, 1], [0.4], 5.0, *synth.gaussian_table(rng, [3], 2))
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)
    G.featurize_points(*a, none, [0, 0], stream=s)
    G.close()
    assert s.query()
