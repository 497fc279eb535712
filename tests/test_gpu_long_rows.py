"""Grids with rows of x too long for the chunk kernels' stages to leave three CTAs on an SM."""
import numpy as np
import pytest

import synth
from test_gpu_parity import W, _spec  # noqa: F401  (W: fixture)
from wri_cases import case, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [628, 632, 634, 1240, 2304])
def test_solves_on_long_rows(W, nx):  # noqa: F811
    """The automatic choice, configurations 18, 22 and 24 and the z-march kernels against complex128 iterates on either
    side of the line (632: boxes; 634 has no boxes; 2304 no chunk kernel): 9 iterations of complex64 round by some
    15 operations each, 9 x 15 x 2^-24 = 8e-6 of the wavefield at the most.  22 and 24 equal 18 bit for bit."""
    G = case(nphys=(nx - 8, 12, 11), npml=4, nsys=2, seed=12, with_data=False)
    G.d = synth.random_complex((len(G.rec_idx),), 3).astype(np.complex64)
    kw = dict(tol=0.0, max_iter=9)
    ref = _spec(W, G, 1)
    W.solve([ref], W.make_opts(dtype=1, kernel=1, **kw))
    exact = ref.u.cpu().numpy()
    got = {}
    for kernel in (0, 1, 2 + 18, 2 + 22, 2 + 24):
        spec = _spec(W, G, 0)
        it, _, _ = W.solve([spec], W.make_opts(dtype=0, kernel=kernel, **kw))
        assert it.cpu().tolist() == [9, 9]
        got[kernel] = spec.u.clone()
        for s in range(2):
            assert rel(spec.u[s].cpu().numpy(), exact[s]) < 8e-6, (kernel, s)
    assert torch.equal(got[2 + 22], got[2 + 18]) and torch.equal(got[2 + 24], got[2 + 18])
