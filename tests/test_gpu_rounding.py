"""Rounding of the FP64 kernels where every term of a kind is equal: flat fields and models."""
import math

import numpy as np
import pytest

import oracle as O
from test_gpu_parity import W, _spec  # noqa: F401  (W: fixture)
from wri_cases import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("nphys,npml,nsys", [((41, 23, 30), 5, 2), ((108, 40, 28), 4, 1), ((30, 9, 8), 0, 2),
                                             ((40, 40, 70), 3, 40)])
def test_constant_field_fp64(W, nphys, npml, nsys):  # noqa: F811
    """A u of a constant field is s_x s_y s_z omega^2 m u off the faces: every difference vanishes, and about two
    roundings of terms as large as u / h^2 are left (the sum of neighbours minus 6 u, and the z + 1 neighbour that is
    added last).  h = 8 makes 1 / h^2 exact, and 1 Hz makes omega^2 m a thousandth of it, so a rounding of the
    diagonal -6 / h^2 or of its product with u (up to 4 / h^2 each) exceeds the bound.  A, A^H and the gradient,
    whose residual is the same stencil; u = 1 + i / 2, so the sums themselves are exact."""
    G = case(nphys=nphys, npml=npml, h=8.0, freq=1.0, nsys=nsys, with_data=False)
    nz, ny, nx = G.spec.shape
    m = 1.0 / np.random.default_rng(5).uniform(1500.0, 3300.0, G.spec.n) ** 2
    spec = _spec(W, G, 1)
    spec.m = torch.from_numpy(m).cuda()
    u = np.full((nsys, G.spec.n), 1.0 + 0.5j)
    om2, ih2 = G.omega ** 2, 1.0 / 64.0
    w = O.stretch_weight(G.spec.shape, 8.0, G.omega, npml, G.v_max, G.pml_R)
    inner = np.zeros(G.spec.shape, bool)
    inner[1:-1, 1:-1, 1:-1] = True
    inner = inner.ravel()
    ut = torch.from_numpy(u).cuda()
    for adjoint in (False, True):
        y = W.apply_A(spec, ut, adjoint=adjoint).cpu().numpy()
        ref = (w.conj() if adjoint else w) * (om2 * m * u[0])
        bound = U * np.abs(w) * abs(u[0, 0]) * (2.5 * ih2 + 16 * om2 * m)
        err = np.abs(y - ref)[:, inner] / bound[inner]
        assert err.max() <= 1.0, (adjoint, err.max())
    spec.u = ut
    spec.d = torch.zeros(len(G.rec_idx), dtype=torch.complex128, device="cuda")
    g, _ = W.gradient([spec], 1, torch.zeros(nsys, dtype=torch.complex128, device="cuda"))
    g = g[0].cpu().numpy().ravel()
    ref = nsys * om2 * np.abs(w) ** 2 * om2 * m * abs(u[0, 0]) ** 2
    bound = U * nsys * om2 * np.abs(w) ** 2 * abs(u[0, 0]) ** 2 * (2.5 * ih2 + (16 + nsys) * om2 * m)
    err = np.abs(g - ref)[inner] / bound[inner]
    assert err.max() <= 1.0, err.max()


@pytest.mark.parametrize("slope", [925311, 571099, 616179])
def test_total_variation_of_equal_cells(W, slope):  # noqa: F811
    """A model with one slope in x, y and z (exact in FP64): all cells and with them nearly all block sums are
    equal, so their additions to the result may all round the same way.  128^3 has 720 blocks; 180 additions
    are off by half a unit of the growing sum each at the most, 90 U in all, and 10 U are left for the sums
    inside.  (An addition per block is off by 115 to 140 U for these slopes.)"""
    n, a, beta = 128, slope * 2.0 ** -50, 1e-9
    i = np.arange(n, dtype=np.float64)
    m = a * (i[:, None, None] + i[None, :, None] + i[None, None, :])
    last = np.ones(n)
    last[-1] = 0.0
    q = np.sqrt(a * a * (last[:, None, None] + last[None, :, None] + last[None, None, :]) + beta * beta)
    ref = math.fsum(q.ravel())
    spec = W.GroupSpec(n, n, n, 0, 10.0, 60.0, 3000.0, None, None, None, None, None, 1.0, None)
    tv, _ = W.tv(spec, torch.from_numpy(m).cuda(), beta)
    assert abs(tv.item() - ref) <= 100 * U * ref, (tv.item() - ref) / ref / U


@pytest.mark.parametrize("nphys,npml", [((150, 21, 20), 0), ((141, 20, 21), 4), ((33, 31, 40), 0)])
def test_sums_of_neighbours_fp64(W, nphys, npml):  # noqa: F811
    """A u and A^H u off the layers for u = 0.9 (1 + i) with random last bits: h = 8 makes 1 / h^2 exact and the exact
    sums are integers.  What rounds are sums of two neighbours below 2 (by 2^-53 at the most, three axes) and of four
    below 4 (by 2^-52); the differences that follow are below 2^-10, so everything else rounds by less than
    2^-8 2^-53 together.  The error of a component is therefore at most 5 2^-53 / h^2 and that.  (Five neighbours in
    one sum round by up to 2^-51 more.)"""
    G = case(nphys=nphys, npml=npml, h=8.0, freq=0.5, nsys=2, with_data=False)
    shape = G.spec.shape
    rng = np.random.default_rng(9)
    ints = np.int64(0.9 * 2 ** 53) + rng.integers(0, 2 ** 40, (2, 2, *shape))  # [system, component, z, y, x]
    spec = _spec(W, G, 1)
    spec.m = torch.full((G.spec.n,), 1.0 / 3000.0 ** 2, dtype=torch.float64, device="cuda")
    vals = ints * 2.0 ** -53
    u = torch.from_numpy(vals[:, 0] + 1j * vals[:, 1]).reshape(2, -1).cuda()
    lap = -6 * ints[..., 1:-1, 1:-1, 1:-1]
    for a in range(3):
        for o in (0, 2):
            cut = [slice(1, -1)] * 3
            cut[a] = slice(o, o + shape[a] - 2)
            lap = lap + ints[(..., *cut)]
    ref = lap * 2.0 ** -59 + G.omega ** 2 / 3000.0 ** 2 * vals[..., 1:-1, 1:-1, 1:-1]
    inner = (..., *[slice(npml, n - 2 - npml) for n in shape])  # nodes npml + 1 .. n - 2 - npml of an axis
    for adjoint in (False, True):
        y = W.apply_A(spec, u, adjoint=adjoint).cpu().numpy().reshape(2, *shape)[..., 1:-1, 1:-1, 1:-1]
        err = np.abs((np.stack([y.real, y.imag], 1) - ref)[inner]).max() * 2.0 ** 59
        assert err <= 5 + 2.0 ** -8, (adjoint, err)
