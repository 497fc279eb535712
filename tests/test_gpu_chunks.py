"""The chunk kernels (linear chunks of the x-y plane, any x extent) at the sizes where they can go wrong:
planes below, at and just past a whole number of chunks, odd and even x extents, grids without a layer and
with a single node between the layers, more z-chunks than one, every right-hand side, both precisions.

Iterate 8 of CGLS, on the chunk kernels and on the z-march kernels, against the oracle's.  Tolerance: 100 u
times the iterate's sensitivity, u = 2^-24 (complex64) or 2^-53: every product with A rounds its 20 or so terms
at u, and the sensitivity is the change of the oracle's own iterate per relative change of A's entries (at
1e-9, in FP64), at least 1.
"""
import numpy as np
import pytest

import oracle as O
import synth
from wri_cases import case, oracle_A, rel, seen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = {0: 2.0 ** -24, 1: 2.0 ** -53}
# physical extents, layer cells
GRIDS = [
    ((8, 8, 12), 4),     # plane 16 x 16 = 256: one chunk exactly
    ((9, 8, 9), 4),      # 17 x 16 = 272: just past it, odd x
    ((5, 6, 5), 0),      # 30 nodes, no layer, odd x
    ((30, 7, 5), 0),     # even x, no layer, odd y
    ((1, 9, 6), 4),      # a single node between the layers (9 x 17 x 14)
    ((34, 13, 1), 3),    # a single plane between the layers, 40 x 19 = 760: three chunks
    ((37, 23, 19), 5),   # odd everything, six chunks
]


@pytest.fixture(scope="module")
def W():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2410_18429_gb300 import wri
    return wri


def _case(grid, mode):
    nphys, npml = grid
    G = case(nphys=tuple(max(v, 3) for v in nphys), npml=npml, nsys=3, nrec=4, seed=17, with_data=False) \
        if min(nphys) < 3 else case(nphys=nphys, npml=npml, nsys=3, nrec=4, seed=17, with_data=False)
    if min(nphys) < 3:  # the generator wants three nodes: rebuild the case on the thin grid by hand
        g = synth.grid(nphys, npml, 10.0)
        r = synth.rng(3)
        v = np.full(g.shape, 2000.0) * (1 + 0.05 * r.standard_normal(g.shape))
        src = np.array([synth.node_index(g, nphys[0] // 2, nphys[1] // 2, nphys[2] // 2) + s for s in (0, 1, g.nx)],
                       np.int64)
        rec = np.array([synth.node_index(g, 0, 0, 0) + 3, synth.node_index(g, 0, 1, 0)], np.int32)
        off, idx = np.arange(4, dtype=np.int32) * 2, np.tile(rec, 3)
        G = synth.Group(g, 12.0, v, src, off, idx, 0.01, 2200.0, alpha=synth.source_weights(3, 18))
    r = synth.rng(5)
    k = int(G.rec_off[-1])
    G.d = (r.standard_normal(k) + 1j * r.standard_normal(k)) * 1e-3
    return G


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("mode", ["free", "known", "rhs", "warm"])
@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g[0])) + f"+{g[1]}")
def test_iterates_match_oracle_and_march(W, grid, mode, dtype):
    from paper_2410_18429_gb300.problem import to_device
    G = _case(grid, mode)
    m, d, alpha = seen(G, dtype == 0)
    n, k = G.spec.n, 8
    cdt = np.complex64 if dtype == 0 else np.complex128
    q = x0 = None
    if mode == "rhs":
        q = synth.random_complex((G.nsys, n), 23).astype(cdt)
    if mode == "warm":
        x0 = synth.random_complex((G.nsys, n), 29).astype(cdt)
    A = oracle_A(G, m)
    got = {}
    for kernel in (0, W.KERNEL_MARCH):
        for zsplit in ((0, 1) if kernel == 0 else (0,)):
            spec = to_device(G, dtype, "cuda", source_free=mode != "known", u=x0)
            if mode == "rhs":
                spec.q = torch.from_numpy(q).cuda()
            it, rr, st = W.solve([spec], W.make_opts(tol=0.0, max_iter=k, dtype=dtype, kernel=kernel, zsplit=zsplit,
                                                     warm_start=mode == "warm"))
            assert it.cpu().tolist() == [k] * G.nsys
            got[kernel, zsplit] = spec.u.cpu().numpy()
    r = synth.rng(31)
    for s in range(G.nsys):
        rec = G.rec_idx[G.rec_off[s]:G.rec_off[s + 1]]
        free = mode in ("free", "warm")
        P = O.restriction(n, rec)
        b = O.rhs(n, G.src[s], d[G.rec_off[s]:G.rec_off[s + 1]], G.lam, alpha[s], mode != "known")
        if mode == "rhs":
            b[:n] = q[s]
        x = None if x0 is None else x0[s].astype(np.complex128)
        ref, _, _ = O.cgls(O.augmented_operator(A, P, G.src[s], G.lam, free), b, tol=0.0, max_iter=k, x0=x)
        A2 = A.copy()
        A2.data = A.data * (1 + 1e-9 * r.standard_normal(A.data.shape))
        off, _, _ = O.cgls(O.augmented_operator(A2, P, G.src[s], G.lam, free), b, tol=0.0, max_iter=k, x0=x)
        tol = 100 * U[dtype] * max(1.0, rel(off, ref) / 1e-9)
        for key, u in got.items():
            assert rel(u[s], ref) < tol, (key, s, rel(u[s], ref), tol)


def test_unaligned_wavefields_and_models(W):
    """complex64 arrays that start 8 bytes past a 16-byte boundary, a model 4 bytes past one: the copies
    round down to the boundary and the kernels index from the remainder."""
    from paper_2410_18429_gb300.problem import to_device
    G = _case(((30, 7, 5), 0), "free")
    ref = to_device(G, 0, "cuda")
    W.solve([ref], W.make_opts(tol=0.0, max_iter=8, dtype=0))
    for nm, nu in ((1, 0), (2, 1), (3, 1)):
        spec = to_device(G, 0, "cuda")
        mb = torch.empty(spec.m.numel() + nm, dtype=torch.float32, device="cuda")
        mb[nm:] = spec.m.reshape(-1)
        spec.m = mb[nm:].view_as(spec.m)
        ub = torch.zeros(spec.u.numel() + nu, dtype=torch.complex64, device="cuda")
        spec.u = ub[nu:].view_as(spec.u)
        W.solve([spec], W.make_opts(tol=0.0, max_iter=8, dtype=0))
        assert rel(spec.u.cpu().numpy(), ref.u.cpu().numpy()) < 1e-5, (nm, nu)


def test_one_systems_nan_stays_its_own(W):
    """A NaN in one system's starting wavefield, next to another system's in memory: the chunk copies of the
    neighbour never carry it over."""
    from paper_2410_18429_gb300.problem import to_device
    G = _case(((9, 8, 9), 4), "warm")
    x0 = synth.random_complex((3, G.spec.n), 29).astype(np.complex64)
    clean = to_device(G, 0, "cuda", u=x0)
    o = W.make_opts(tol=0.0, max_iter=6, dtype=0, warm_start=True)
    W.solve([clean], o)
    x0[1, 0] = x0[1, -1] = np.nan
    spec = to_device(G, 0, "cuda", u=x0)
    _, _, st = W.solve([spec], o)
    st = st.cpu().tolist()
    assert st[1] == W.SYS_NONFINITE and st[0] == st[2] == W.SYS_MAXITER
    for s in (0, 2):
        assert np.array_equal(spec.u[s].cpu().numpy(), clean.u[s].cpu().numpy())


def test_complex64_gradient_scales_exactly_and_keeps_nan_at_its_nodes(W):
    """The complex64 gradient widens its float terms in integer arithmetic: scaling u by 2^-30 scales every
    term, so the gradient, by exactly 2^-60; a NaN (which takes the conversion instruction, as subnormals and
    infinities do) stays at its node's and its neighbours' terms."""
    from paper_2410_18429_gb300.problem import to_device
    G = _case(((37, 23, 19), 5), "free")
    G.d[:] = 0
    n = G.spec.n
    u0 = (synth.random_complex((3, n), 41) * 1e-3).astype(np.complex64)

    def grad(scale, bad=None):
        u = (u0 * np.float32(scale)).astype(np.complex64)
        if bad is not None:
            u[1, bad] = np.nan
        spec = to_device(G, 0, "cuda", u=u)
        a = torch.zeros(3, dtype=torch.complex128, device="cuda")
        (g,), _ = W.gradient([spec], 0, a)
        return g.cpu().numpy().ravel()

    g1 = grad(1.0)
    assert np.array_equal(grad(2.0 ** -30), g1 * 2.0 ** -60)
    bad = n // 2 + 5
    gn = grad(1.0, bad)
    nx, pl = G.spec.nx, G.spec.nx * G.spec.ny
    touched = {bad, bad - 1, bad + 1, bad - nx, bad + nx, bad - pl, bad + pl}
    assert set(np.flatnonzero(np.isnan(gn))) == touched
    keep = np.setdiff1d(np.arange(n), sorted(touched))
    assert np.array_equal(gn[keep], g1[keep])
