"""Refined solves: a general right-hand side q (A u = q together with the data), and the boxes' phases."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

import oracle as O
import synth
from test_gpu_parity import W, _exact, _spec  # noqa: F401  (W: fixture)
from wri_cases import case, oracle_A, rel, seen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("nphys,kernel", [((15, 11, 9), 0), ((18, 11, 9), 0), ((18, 11, 9), 11),
                                          ((18, 11, 9), 19), ((15, 11, 9), 1)])
def test_refined_general_right_hand_side_matches_exact(W, nphys, kernel, warm):  # noqa: F811
    """FP64 refinement of min ||A u - q||^2 + lambda^2 ||P u - d||^2 from a cold and from a warm start (odd and even
    x extent on the chunk kernels, the boxes of configurations 9 and 17, z-march): the FP64 wavefield against the sparse
    LU solution, with the error that a normal residual of 1e-10 allows in the other refinement tests."""
    G = case(nphys=nphys, npml=3, nsys=2, freq=15.0)
    m, d, _ = seen(G, True)
    n = G.spec.n
    q = (synth.random_complex((G.nsys, n), 9) * 1e-3).astype(np.complex64)
    x0 = (synth.random_complex((G.nsys, n), 11) * 1e-3).astype(np.complex64) if warm else None
    spec = _spec(W, G, 0, u=x0)
    spec.q = torch.from_numpy(q).cuda()
    spec.u64 = torch.full((G.nsys, n), np.nan, dtype=torch.complex128, device="cuda")
    it, rr, st = W.solve([spec], W.make_opts(tol=1e-3, max_iter=200000, dtype=0, max_refine=12, refine_tol=1e-10,
                                             inner_tol=1e-2, kernel=kernel, warm_start=warm))
    assert st.cpu().tolist() == [W.SYS_OK] * G.nsys, (st, rr, it)
    assert 0 < float(rr.min()) and float(rr.max()) <= 1e-10
    lu = spla.splu(oracle_A(G, m).tocsc())
    u = spec.u64.cpu().numpy()
    for s in range(G.nsys):
        rec = G.rec_idx[G.rec_off[s]:G.rec_off[s + 1]]
        u0 = lu.solve(q[s].astype(np.complex128))  # the rest is a problem without a right-hand side
        w = O.solve_dataspace(lu, n, G.src[s], rec, d[G.rec_off[s]:G.rec_off[s + 1]] - u0[rec], G.lam, 0.0, False)
        assert rel(u[s], u0 + w) < 1e-8
    assert torch.equal(spec.u.to(torch.complex128), spec.u64.to(torch.complex64).to(torch.complex128))


@pytest.mark.parametrize("cfg", [9, 12, 17])
@pytest.mark.parametrize("source_free", [True, False])
def test_refinement_on_boxes_matches_exact(W, source_free, cfg):  # noqa: F811
    """Refined solves whose inner phases run on the TMA boxes (phase 2 adds S^H r64), among the candidates of
    wri_autotune: as test_refinement_on_tma_phases_matches_exact, which runs on the chunk kernels."""
    G = case(nphys=(16, 11, 9), npml=4, nsys=2, freq=15.0)
    m, d, _ = seen(G, True)
    spec = _spec(W, G, 0, source_free)
    spec.u64 = torch.zeros(G.nsys, G.spec.n, dtype=torch.complex128, device="cuda")
    it, rr, st = W.solve([spec], W.make_opts(tol=1e-3, max_iter=200000, dtype=0, max_refine=12, refine_tol=1e-10,
                                             inner_tol=1e-2, kernel=W.KERNEL_TMA(cfg)))
    assert st.cpu().tolist() == [W.SYS_OK] * 2, (st, rr, it)
    for s in range(2):
        assert rel(spec.u64[s].cpu().numpy(), _exact(G, m, d, source_free, s)) < 1e-8
