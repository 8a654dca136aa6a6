"""Gradients of a handle whose batches grow from call to call, each buffer of it
moving into memory that others filled before, to the bit of a fresh handle's."""
import ctypes as C

import numpy as np
import pytest

from paper_2303_12980_gb300 import synth
from paper_2303_12980_gb300.binding import load_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    return t


def _dirty(n_bytes):
    """Blocks of device memory beside the library's own, filled with ones and
    handed back (a block that holds no other comes back cleared)."""
    L = load_library()
    blocks = []
    for size in [n_bytes] * 3 + [max(n_bytes // 8, 256)] * 24:
        p = C.c_void_p()
        assert L.cudaMalloc(C.byref(p), C.c_size_t(size)) == 0 and L.cudaMemset(p, 255, C.c_size_t(size)) == 0
        blocks.append(p)
    for p in blocks:
        assert L.cudaFree(p) == 0


@pytest.mark.parametrize("n0,n1,step", [(2, 200, 1.2), (20, 3000, 1.2), (2000, 100_000, 1.3)])
def test_gradients_of_growing_batches(torch, n0, n1, step):
    from paper_2303_12980_gb300.binding import GMPFeaturizer
    rng = np.random.default_rng(n0)
    table = synth.gaussian_table(rng, [3, 4], 2)

    def call(F, n):
        r = np.random.default_rng(n)
        S = n // 2
        pos = torch.from_numpy(r.uniform(0, 1.5, (2 * S, 3))).cuda()
        sp = torch.from_numpy(r.integers(0, 2, 2 * S).astype(np.int32)).cuda()
        g = torch.from_numpy(synth.upstream_gradient(2 * S, F.num_features, seed=n)).cuda()
        _, gp = F.featurize_vjp(pos, sp, np.arange(S + 1) * 2, np.zeros((S, 3, 3)), np.zeros((S, 3), np.uint8), g)
        return gp.cpu()

    new = lambda: GMPFeaturizer([0, 1], [0.4, 0.8], 4.0, *table)
    F, n = new(), n0
    while n <= n1:
        _dirty(288 * n)
        got = call(F, n)
        assert torch.isfinite(got).all() and torch.equal(got, call(new(), n)), n
        n = int(n * step) + 2
