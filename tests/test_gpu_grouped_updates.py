"""Iterate updates of the chunk kernels grouped over several iterations."""
import numpy as np
import pytest

from test_gpu_parity import W, _spec  # noqa: F401  (W: fixture)
from wri_cases import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("nphys", [(36, 13, 10), (29, 12, 11)])
def test_grouped_updates_equal_single_updates(W, nphys, dtype):  # noqa: F811
    """Configurations 22 and 24 (x updated every second and fourth iteration) against 18 (every iteration) on an even
    and an odd x extent: wavefields, residuals and counts bit for bit after 1 to 9 iterations (every number of
    pending steps), in loop bodies that hold all iterations and in shorter ones, and for systems that stop by their
    tolerance at different iterations."""
    G = case(nphys=nphys, npml=4, nsys=3, seed=12)

    def run(cfg, **kw):
        spec = _spec(W, G, dtype)
        it, rr, st = W.solve([spec], W.make_opts(dtype=dtype, kernel=W.KERNEL_TMA(cfg), **kw))
        return [t.cpu().numpy() for t in (spec.u, it, rr, st)]

    cases = [dict(tol=0.0, max_iter=k, poll_every=p) for k in range(1, 10) for p in (0, 4)]
    cases.append(dict(tol=1e-2, max_iter=100000))
    for kw in cases:
        single = run(18, **kw)
        for cfg in (22, 24):
            for a, b in zip(run(cfg, **kw), single):
                assert np.array_equal(a, b), (cfg, kw)
    assert single[3].tolist() == [W.SYS_OK] * 3 and len(set((single[1] % 4).tolist())) > 1, single[1]


def test_grouped_updates_of_refined_solves_on_an_odd_extent(W):  # noqa: F811
    """The same over several outer steps of a refined solve, with and without an FP64 array of the caller's."""
    G = case(nphys=(29, 12, 11), npml=4, nsys=3, seed=12)
    out = []
    for cfg, wide in ((18, True), (24, True), (22, False), (24, False)):
        spec = _spec(W, G, 0)
        if wide:
            spec.u64 = torch.zeros(G.nsys, G.spec.n, dtype=torch.complex128, device="cuda")
        it, rr, st = W.solve([spec], W.make_opts(dtype=0, tol=1e-3, max_iter=37, max_refine=3, refine_tol=1e-12,
                                                 inner_tol=1e-12, kernel=W.KERNEL_TMA(cfg)))
        assert it.cpu().tolist() == [3 * 37] * 3, it
        out.append([spec.u.clone(), rr, it])
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(o, out[0]))
