"""The tensor-core FP64 element kernel on elements whose values differ by many
orders of magnitude, at the degrees where it follows every line (N = 3, 15):
each contraction is accurate to its own line, as floating-point arithmetic is,
not to the element's largest value.

The bound: with eps = 2^-53, a contraction of a line is off by at most
c eps rowsum|D| max|line| and the metric step and the sums by a few eps of their
terms. B below adds these with c = 1 in 64 bits; the kernel's own share of c is
below 1/4 (a value is rounded to 2^-56 of its line's largest), the conversion of
a sum to a double 1/2 and the remaining sums a few eps of terms that B holds, so
4 B covers it. A grid per element is off by up to 1e8 B here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb, inputs  # noqa: E402
from test_gpu_tc_degrees import _dev, _extended  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def _bound(m, N, x, lam):
    n, eps = N + 1, 2.0 ** -53
    L = np.polynomial.legendre.Legendre.basis(N)
    xi = np.concatenate([[-1.0], np.sort(L.deriv().roots().real), [1.0]])
    P = L(xi)
    D = np.array([[0.0 if i == j else P[i] / (P[j] * (xi[i] - xi[j])) for j in range(n)] for i in range(n)])
    D[0, 0] = D[N, N] = N * (N + 1) / 4
    D = np.abs(D)
    G = np.abs(m.geo()).reshape(m.E, n, 7, n, n)
    l2g = m.l2g().reshape(m.E, n, n, n)
    u = np.abs(np.where(l2g >= 0, x[np.maximum(l2g, 0)], 0.0))
    ax = (3, 2, 1)  # r, s, t

    def lines(w, M):  # rowsum(M)_i max of the line, per node
        return [np.broadcast_to(w[d].max(a, keepdims=True), u.shape) *
                M.sum(1).reshape([n if q == a else 1 for q in range(4)]) for d, a in enumerate(ax)]
    g = lines([u] * 3, D)
    # |v|: at most |G| g, its error eps times the same
    v = [G[:, :, c[0]] * g[0] + G[:, :, c[1]] * g[1] + G[:, :, c[2]] * g[2] for c in ((0, 1, 2), (1, 3, 4), (2, 4, 5))]
    y = sum(lines(v, D.T))  # of eps |v| (error carried through) and of the second contraction's own error
    out = lam * np.abs(x)
    np.add.at(out, l2g[l2g >= 0], 2.0 * y[l2g >= 0])
    return eps * out


@pytest.mark.parametrize("N,dims", [(3, (4, 3, 5)), (15, (2, 2, 2))])
@pytest.mark.parametrize("kind", ["one_large", "decades", "layer"])
@pytest.mark.parametrize("variant", hb.VARIANTS_TC)
@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="needs an extended long double")
def test_tc_graded_element(N, dims, kind, variant):
    m = hb.Mesh(*dims, N, perturb=0.1, seed=1, faces=0x15, fp32=False)
    rng = np.random.Generator(np.random.PCG64(N))
    x = inputs.random_vector(m.n_global, seed=21)
    if kind == "one_large":  # one node in the inside of some elements 1e8 times the others
        l2g = m.l2g().reshape(m.E, N + 1, N + 1, N + 1)
        x[l2g[::2, 1, N - 1, 1]] *= 1e8
    elif kind == "decades":
        x *= 10.0 ** rng.uniform(-6, 6, m.n_global)
    else:  # values that fall by 1e10 over the box
        x *= 10.0 ** -(10.0 * np.arange(m.n_global) / m.n_global)
    hb.hb_set_kernel_variant(m.handle, hb.HB_F64, variant)
    y = m.apply_A(_dev(x), lam=0.1).cpu().numpy()
    ratio = np.abs((y - _extended(m, N, x, 0.1)).astype(float)) / _bound(m, N, x, 0.1)
    print(N, kind, variant, ratio.max())
    assert ratio.max() <= 4.0
    m.close()
