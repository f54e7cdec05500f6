"""The state read back in key order (a radix sort on the device) against the
unordered device copy of the same state, sorted here: the same keys, amplitudes
and sigma, at the edges of the sort's tiles of 4,096, with one determinant, and
with keys that fill one word, half of one and two."""
import ctypes

import numpy as np
import pytest

from paper_2301_05726_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [False, True])
@pytest.mark.parametrize("n,keep", [(10, 1), (10, 4095), (10, 4096), (10, 4097), (32, 20000), (33, 4097), (40, 9000)])
def test_matches_the_unordered_copy(n, keep, sigma):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05726_gb300 import build
    build.build()
    from paper_2301_05726_gb300.api import UCCContext
    p = synth.make_problem(5, n, 4, 4, 0.2, name="sorted").prefix(200)
    p.n_max = p.n_cut = keep
    ctx = UCCContext(p)
    ctx.apply()
    if sigma:
        ctx.energy()
    got = ctx.wavefunction(with_sigma=sigma)
    count = len(got[1])
    assert count == keep
    words = ctx.key_words
    dk = torch.zeros(count * words, dtype=torch.int64, device="cuda")
    da, ds = (torch.zeros(count, dtype=torch.float64, device="cuda") for _ in range(2))
    size = ctypes.c_size_t()
    assert ctx.lib.ucc_get_wavefunction(ctx.handle, count, ctypes.byref(size), ctypes.c_void_p(dk.data_ptr()),
                                        ctypes.c_void_p(da.data_ptr()),
                                        ctypes.c_void_p(ds.data_ptr()) if sigma else None, 1) == 0
    keys = dk.cpu().numpy().view(np.uint64).reshape(count, words)
    order = np.lexsort(tuple(keys.T))
    assert size.value == count and np.array_equal(got[0].reshape(count, words), keys[order])
    assert np.array_equal(got[1], da.cpu().numpy()[order])
    if sigma:
        assert np.array_equal(got[2], ds.cpu().numpy()[order])
