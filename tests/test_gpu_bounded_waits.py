"""Bounded waits of the copy pipelines: time-outs are reported and leave the context usable."""
import pytest

from test_gpu_parity import W, _spec  # noqa: F401  (W: fixture)
from wri_cases import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit_us", [1, 1000])
@pytest.mark.parametrize("dtype,cfg", [(0, 24), (1, 24), (0, 9), (0, 17)])
def test_time_out_of_items_shorter_than_the_ring(W, dtype, cfg, limit_us):  # noqa: F811
    """One plane per work item: the copy warp of block 0 issues its last copy without waiting for a stage, so
    only the wait before it leaves keeps the copies behind the withheld one inside the CTA's lifetime, also
    with a limit shorter than a copy takes.  The call returns WRI_ECUDA and the next solve is unharmed."""
    G = case(nphys=(36, 13, 10), npml=4, nsys=3)
    nz, k = 18, 6
    kw = dict(tol=0.0, max_iter=k, dtype=dtype, kernel=W.KERNEL_TMA(cfg), zsplit=nz)
    ref = _spec(W, G, dtype)
    W.solve([ref], W.make_opts(**kw))
    for withhold in (1, 2):
        bad = _spec(W, G, dtype)
        with pytest.raises(W.WriError) as e:
            W.solve([bad], W.make_opts(wait_limit_us=limit_us, test_withhold=withhold, **kw))
        assert e.value.code == W.ECUDA
        torch.cuda.synchronize()
        again = _spec(W, G, dtype)
        it, _, _ = W.solve([again], W.make_opts(**kw))
        assert it.cpu().tolist() == [k] * 3
        assert torch.equal(again.u, ref.u)


def test_time_out_of_a_refined_solve_in_its_first_pass(W):  # noqa: F811
    """A general right-hand side under refinement, one system, 24 x 43 x 43: the complex64 pass that forms S^H b
    has two planes per work item and the FP64 passes one, so of all passes before the first iteration only
    this one reaches the third fill of block 0.  Its system never starts, and the call must not report it as
    solved: WRI_ECUDA, and the next solve is unharmed."""
    G = case(nphys=(18, 37, 37), npml=3, nsys=1)
    g = torch.Generator().manual_seed(3)
    q = torch.randn(1, G.spec.n, dtype=torch.complex64, generator=g)
    kw = dict(tol=1e-3, max_iter=12, dtype=0, max_refine=1, refine_tol=1e-12, inner_tol=1e-3)

    def spec():
        s = _spec(W, G, 0)
        s.q = q.cuda()
        s.u64 = torch.zeros(1, G.spec.n, dtype=torch.complex128, device="cuda")
        return s

    ref = spec()
    it, _, _ = W.solve([ref], W.make_opts(**kw))
    assert it.cpu().tolist() == [12]
    with pytest.raises(W.WriError) as e:
        W.solve([spec()], W.make_opts(wait_limit_us=1000, test_withhold=3, **kw))
    assert e.value.code == W.ECUDA
    torch.cuda.synchronize()
    again = spec()
    W.solve([again], W.make_opts(**kw))
    assert torch.equal(again.u64, ref.u64)
