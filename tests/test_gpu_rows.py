"""The rows of Z^T and the FP32 factors that mesh set-up forms directly: CSR
arrays against a plain construction from the node map (every face mask, single
elements, N = 1), the lumped mass against the factors, and the integer rounding
of the FP32 copies against numpy's, zeros and tiny values included."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


class _View:
    def __init__(self, ptr, n, kind):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind, "data": (ptr, False), "version": 2}


def _host(ptr, n, kind):
    return torch.as_tensor(_View(ptr, n, kind), device="cuda").cpu().numpy() if n else np.zeros(0, kind)


@pytest.mark.parametrize("dims,N", [((1, 1, 1), 1), ((1, 1, 1), 2), ((2, 1, 3), 1), ((3, 2, 2), 3), ((1, 4, 2), 5),
                                    ((2, 2, 2), 8), ((5, 1, 1), 15), ((7, 9, 11), 2),
                                    ((700, 1, 2), 2)])
@pytest.mark.parametrize("faces", [0x3F, 0x00, 0x15, 0x2A, 0x07])
@pytest.mark.parametrize("perturb", [0.0, 0.2])
def test_rows_and_copies(dims, N, faces, perturb):
    m = hb.Mesh(*dims, N, perturb=perturb, seed=4, faces=faces, fp32=True)
    i = m.info
    l2g = m.l2g()
    at = np.nonzero(l2g >= 0)[0]
    assert i.nnz == at.size and m.n_global == (l2g.max() + 1 if at.size else 0)
    order = at[np.argsort(l2g[at], kind="stable")]
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(l2g[at], minlength=m.n_global))]).astype(np.int32)
    assert np.array_equal(_host(i.csr_rowptr, m.n_global + 1, "<i4"), rowptr)
    assert np.array_equal(_host(i.csr_cols, i.nnz, "<i4"), order)
    geo = m.geo()
    assert np.array_equal(_host(i.geo32, geo.size, "<f4"), geo.astype(np.float32))
    # A 1 with mass screening and D 1 = 0: the lumped mass, summed over each row (and the surface rows)
    n = N + 1
    jw = geo.reshape(m.E, n, 7, n, n)[:, :, 6].reshape(-1)
    if m.n_global and faces == 0:
        mass = np.zeros(m.n_global)
        np.add.at(mass, l2g[order], jw[order])
        for v in (0, 3, 67):
            hb.hb_set_kernel_variant(m.handle, hb.HB_F64, v)
            y = m.apply_A(torch.ones(m.n_global, dtype=torch.float64, device="cuda"), lam=1.0, screen=1).cpu().numpy()
            assert np.abs(y - mass).max() <= 1e-12 * np.abs(geo).max() * N * N
    m.close()
