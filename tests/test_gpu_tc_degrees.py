"""The tensor-core FP64 element kernel at each degree it is built for: against
the oracle at the FP64 bars, on element counts around its tiles (16 elements
at N = 3, 2 at N = 7, 1 at N = 15), and against an evaluation in extended
precision, where its error is no larger than the FP64 pencil kernel's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import oracle as orc  # noqa: E402
from paper_2202_12477_gb300 import hb, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("dims,N", [((1, 1, 1), 3), ((5, 3, 1), 3), ((4, 4, 1), 3), ((17, 1, 1), 3), ((7, 6, 5), 3),
                                    ((1, 1, 1), 15), ((2, 1, 1), 15), ((3, 2, 2), 15), ((3, 3, 1), 7)])
@pytest.mark.parametrize("screen,lam,faces", [(0, 0.1, 0x3F), (1, 0.7, 0x15)])
@pytest.mark.parametrize("variant", hb.VARIANTS_TC)
def test_tc_degrees_match_oracle(dims, N, screen, lam, faces, variant):
    m = hb.Mesh(*dims, N, perturb=0.15, seed=sum(dims), faces=faces, fp32=False)
    o = orc.Mesh(*dims, N, rho=0.15, seed=sum(dims), faces=faces)
    hb.hb_set_kernel_variant(m.handle, hb.HB_F64, variant)
    x = inputs.random_vector(m.n_global, seed=77)
    for scale in (1.0, 1e-200, 1e200):
        y = m.apply_A(_dev(x * scale), lam=lam, screen=screen).cpu().numpy() / scale
        y_or = o.apply_A(x, lam, screen)
        assert np.linalg.norm(y - y_or) <= 1e-12 * np.linalg.norm(y_or)
        assert np.abs(y - y_or).max() <= 1e-12 * np.abs(y_or).max()
    b = m.rhs(kind=0, seed=2)
    hb.lib().hb_set_cg_fused(m.handle, 1)
    xs, res = m.cg(b, lam=1.0, max_it=15)  # x.y partials of the element kernel
    x_or, *_ = o.cg(b.cpu().numpy(), 1.0, rtol=0.0, max_it=15)
    assert np.linalg.norm(xs.cpu().numpy() - x_or) <= 1e-12 * np.linalg.norm(x_or)
    m.close()


@pytest.mark.parametrize("N", hb.TC_DEGREES)
def test_tc_nonfinite(N):
    m = hb.Mesh(3, 2, 2, N, perturb=0.1, seed=5, fp32=False)
    hb.hb_set_kernel_variant(m.handle, hb.HB_F64, hb.HB_VARIANT_TC)
    x = inputs.random_vector(m.n_global, seed=43)
    y0 = m.apply_A(_dev(x), lam=0.1).cpu().numpy()
    l2g = m.l2g().reshape(m.E, -1)
    for bad in (np.nan, np.inf):
        g = m.n_global // 2
        xb = x.copy()
        xb[g] = bad
        y = m.apply_A(_dev(xb), lam=0.1).cpu().numpy()
        touched = np.unique(l2g[(l2g == g).any(axis=1)])
        far = np.setdiff1d(np.arange(m.n_global), touched)
        assert np.isnan(y[touched[touched >= 0]]).all() and np.array_equal(y[far], y0[far])
    m.close()


def _extended(m, N, x, lam):
    """A x in extended precision from the mesh's own (rounded) factors; D from the nodes in long double."""
    L = np.longdouble
    n = N + 1
    xi = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.Legendre.basis(N).deriv().roots().real), [1.0]]).astype(L)

    def leg(z):
        a, b, da, db = L(1) + 0 * z, z, 0 * z, L(1) + 0 * z
        for k in range(2, N + 1):
            a, b, da, db = b, ((2 * k - 1) * z * b - (k - 1) * a) / L(k), db, da + (2 * k - 1) * b
        return a, b, db
    for _ in range(4):  # Newton on N (P_{N-1} - x P_N), derivative -N (N + 1) P_N
        a, b, _d = leg(xi[1:-1])
        xi[1:-1] += (a - xi[1:-1] * b) / ((N + 1) * b)
    xi = (xi - xi[::-1]) / 2
    P = leg(xi)[1]
    D = np.zeros((n, n), dtype=L)
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = P[i] / (P[j] * (xi[i] - xi[j]))
    D[0, 0], D[N, N] = -L(N * (N + 1)) / 4, L(N * (N + 1)) / 4
    G = m.geo().reshape(m.E, n, 7, n, n).astype(L)
    l2g = m.l2g().reshape(m.E, n, n, n)
    u = np.where(l2g >= 0, x[np.maximum(l2g, 0)], 0.0).astype(L)
    ur, us, ut = (np.einsum(s, D, u) for s in ("im,ekjm->ekji", "jm,ekmi->ekji", "km,emji->ekji"))
    v = [G[:, :, c[0]] * ur + G[:, :, c[1]] * us + G[:, :, c[2]] * ut for c in ((0, 1, 2), (1, 3, 4), (2, 4, 5))]
    yl = sum(np.einsum(s, D, w) for s, w in zip(("mi,ekjm->ekji", "mj,ekmi->ekji", "mk,emji->ekji"), v))
    y = lam * x.astype(L)
    np.add.at(y, l2g[l2g >= 0], yl[l2g >= 0])
    return y


@pytest.mark.parametrize("N,dims", [(3, (6, 5, 7)), (7, (4, 4, 4)), (15, (3, 2, 2))])
@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="needs an extended long double")
def test_tc_error_no_larger_than_pencil(N, dims):
    m = hb.Mesh(*dims, N, perturb=0.1, seed=1, fp32=False)
    for kind in ("uniform", "normal"):
        x = inputs.random_vector(m.n_global, seed=21, kind=kind)
        ref = _extended(m, N, x, 0.1)
        err = {}
        for v in (3, hb.HB_VARIANT_TC):
            hb.hb_set_kernel_variant(m.handle, hb.HB_F64, v)
            y = m.apply_A(_dev(x), lam=0.1).cpu().numpy()
            err[v] = float(np.sqrt(((y - ref) ** 2).sum() / (ref ** 2).sum()))
        print(N, kind, err)
        assert err[hb.HB_VARIANT_TC] <= err[3]
    m.close()
