"""The element kernel that spreads one element over a cluster of blocks (small
FP64 and double-float meshes, double-float from N = 11 on): value for value
the result of the other pencil variants, on one, two and four blocks per
element, even and odd lines; and the fused CG built on it against the launched
kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


# four blocks per element (few elements, high degree), two, one, the base shape
@pytest.mark.parametrize("dims,N", [((1, 1, 1), 2), ((2, 1, 1), 15), ((3, 2, 1), 14), ((2, 2, 2), 11), ((5, 2, 4), 9),
                                    ((4, 4, 4), 8), ((19, 2, 2), 7), ((7, 11, 1), 7), ((3, 3, 3), 3), ((5, 5, 5), 4),
                                    ((6, 7, 8), 6), ((10, 9, 8), 5), ((8, 19, 1), 10), ((6, 5, 6), 13), ((3, 7, 8), 15),
                                    ((7, 7, 7), 12)])
@pytest.mark.parametrize("prec", [hb.HB_F64, hb.HB_F64X])
def test_split_equals_other_variants(dims, N, prec):
    m = hb.Mesh(*dims, N, perturb=0.15, seed=N, faces=0x15, fp32=False)
    x = torch.from_numpy(inputs.random_vector(m.n_global, seed=N + 1)).cuda()
    for screen, lam in [(0, 0.1), (1, 0.6)]:
        y = {}
        for v in (3, 67):
            hb.hb_set_kernel_variant(m.handle, prec, v)
            y[v] = m.apply_A(x, lam=lam, screen=screen, prec=prec).cpu().numpy()
        assert np.array_equal(y[3], y[67])
    # the partials of x.y (every block of a cluster has one) through CG: the
    # same iterates as with the other variant, to the rounding of the sums
    b = m.rhs(kind=0, seed=3)
    hb.lib().hb_set_cg_fused(m.handle, 1)
    xs = {}
    for v in (3, 67):
        hb.hb_set_kernel_variant(m.handle, prec, v)
        xs[v] = m.cg(b, lam=0.5, max_it=12, prec=prec)[0].cpu().numpy()
    assert np.linalg.norm(xs[3] - xs[67]) <= 1e-12 * np.linalg.norm(xs[67])
    m.close()


@pytest.mark.parametrize("dims,N", [((1, 1, 1), 2), ((2, 2, 1), 1), ((3, 3, 3), 7), ((4, 4, 4), 7), ((6, 6, 6), 7),
                                    ((3, 3, 3), 15), ((4, 3, 5), 9), ((5, 5, 4), 12), ((2, 2, 2), 8)])
@pytest.mark.parametrize("screen", [0, 1])
def test_fused_cg_equals_launched(dims, N, screen):
    m = hb.Mesh(*dims, N, perturb=0.1, seed=1, faces=0x07 if N < 3 else 0x3F, fp32=False)
    b = m.rhs(kind=0, seed=5)
    x0 = torch.from_numpy(inputs.random_vector(m.n_global, seed=8)).cuda()
    got = {}
    for mode in (1, 2):
        hb.lib().hb_set_cg_fused(m.handle, mode)
        x, r = m.cg(b, x0.clone(), lam=0.3, screen=screen, max_it=min(25, m.n_global))
        assert r.status == hb.HB_OK
        got[mode] = x.cpu().numpy()
        # bitwise repeatable, stopped on the tolerance, and zero iterations
        assert np.array_equal(got[mode], m.cg(b, x0.clone(), lam=0.3, screen=screen,
                                              max_it=min(25, m.n_global))[0].cpu().numpy())
    assert np.linalg.norm(got[1] - got[2]) <= 1e-12 * np.linalg.norm(got[1])
    xt, rt = m.cg(b, x0.clone(), lam=0.3, screen=screen, rtol=1e-9, max_it=3000)
    assert rt.status == hb.HB_OK and rt.rel_res <= 1e-9
    xz, rz = m.cg(b, x0.clone(), lam=0.3, screen=screen, max_it=0)
    assert rz.iters == 0 and torch.equal(xz, x0)
    m.close()


@pytest.mark.parametrize("dims,N,prec", [((80, 81, 80), 3, hb.HB_F32), ((80, 81, 80), 3, hb.HB_F64),
                                         ((40, 39, 41), 7, hb.HB_F64X), ((20, 20, 19), 15, hb.HB_F32)])
def test_large_Ax_by_lattice_equals_surface_rows(dims, N, prec):
    """From 30 million local nodes on A x alone takes Z^T by the lattice: the
    same values as through the surface rows, which the dot modes (CG) keep."""
    m = hb.Mesh(*dims, N, perturb=0.1, seed=2, faces=0x15, fp32=prec == hb.HB_F32)
    assert m.n_local >= 30_000_000
    dt = torch.float32 if prec == hb.HB_F32 else torch.float64
    x = torch.from_numpy(inputs.random_vector(m.n_global, seed=6)).to(dt).cuda()
    y = {}
    for v in (3, 67):
        hb.hb_set_kernel_variant(m.handle, prec, v)
        y[v] = m.apply_A(x, lam=0.4, screen=1, prec=prec)
    assert torch.equal(y[3], y[67])
    m.close()
