"""Reuse of the captured iterations from call to call."""
import time

import pytest

from test_gpu_parity import W, _spec  # noqa: F401  (W: fixture)
from wri_cases import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_new_fp64_arrays_do_not_recapture_the_iterations(W):  # noqa: F811
    """The iterations of a refined solve never touch its FP64 solution, so a call with another u64 array replays the
    graph of the call before: the fastest of 30 calls with new arrays within 1.2 of the fastest with one array (with a
    capture in each they take 1.4 times as long), in one of three attempts."""
    G = case(nphys=(28, 12, 10), npml=4, nsys=2)
    spec = _spec(W, G, 0)
    opts = W.make_opts(tol=1e-3, max_iter=4, dtype=0, max_refine=1, refine_tol=1e-12, inner_tol=1e-3)
    arrays = [torch.zeros(2, G.spec.n, dtype=torch.complex128, device="cuda") for _ in range(31)]
    work = torch.empty(W.workspace_size([spec], opts), dtype=torch.uint8, device="cuda")

    def seconds(a):
        spec.u64 = a
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        W.solve([spec], opts, workspace=work)
        torch.cuda.synchronize()
        return time.perf_counter() - t0

    ratios = []
    for attempt in range(3):
        for _ in range(5):
            seconds(arrays[0])
        one = min(seconds(arrays[0]) for _ in range(30))
        ratios.append(min(seconds(a) for a in arrays[1:]) / one)
        if ratios[-1] < 1.2:
            return
    raise AssertionError(ratios)
