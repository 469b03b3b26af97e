"""mmp_demag_noalloc over the transform engines it chooses from (block passes, one, two and four classes of
kx, two of ky) against the context path, and captured into a CUDA graph: the replay on other inputs gives
bitwise what direct calls give."""
import numpy as np
import pytest

from test_zz_no_alloc import _context_demag

pytestmark = pytest.mark.gpu

CELL = (2e-9, 2.5e-9, 1.5e-9)
MS = 8e5


def _M(seed, shape):
    import torch
    from inputs import random_unit_vectors
    return torch.from_numpy(random_unit_vectors(seed, shape) * np.float32(MS)).cuda()


@pytest.mark.parametrize("shape", [(20, 18, 2), (33, 27, 5), (600, 9, 1), (1000, 7, 1), (1100, 10, 1), (2046, 3, 1),
                                   (9, 700, 2), (40, 900, 1)])
def test_noalloc_matches_context_path(shape):
    import torch
    import paper_2411_18194_gb300 as pkg
    from inputs import MU0
    for seed in (3, 4):
        M = _M(seed, shape)
        B = torch.full_like(M, float("nan"))
        pkg.demag_noalloc(shape, CELL, M, B)
        torch.cuda.synchronize()
        assert np.abs(B.cpu().numpy() - _context_demag(shape, CELL, M)).max() <= 1e-5 * MU0 * MS


@pytest.mark.parametrize("shape", [(64, 48, 1), (1100, 10, 1), (20, 18, 2)])
def test_noalloc_captured_equals_direct(shape):
    import torch
    import paper_2411_18194_gb300 as pkg
    s = torch.cuda.Stream()
    M = _M(5, shape)
    B, C = torch.empty_like(M), torch.empty_like(M)
    s.wait_stream(torch.cuda.current_stream())
    pkg.demag_noalloc(shape, CELL, M, B, stream=s)     # the set-up is not captured
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        pkg.demag_noalloc(shape, CELL, M, B, stream=torch.cuda.current_stream())
        pkg.demag_noalloc(shape, CELL, B, C, stream=torch.cuda.current_stream())
    for seed in (6, 7):
        M.copy_(_M(seed, shape))
        g.replay()
        torch.cuda.synchronize()
        b, c = B.clone(), C.clone()
        pkg.demag_noalloc(shape, CELL, M, B)
        pkg.demag_noalloc(shape, CELL, B, C)
        torch.cuda.synchronize()
        assert torch.equal(B, b) and torch.equal(C, c)
