"""A kernel that runs in clusters and finds itself outside the shape it was
launched for touches no other block: NaN results and an error status, and the
context stays usable."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def test_cluster_shape_is_checked():
    assert hb.hb_selftest_cluster(True) == hb.HB_OK
    assert hb.hb_selftest_cluster(False) == hb.HB_ERR_CUDA
    with pytest.raises(hb.HBError):
        hb.hb_selftest_cluster(2)
    m = hb.Mesh(3, 3, 3, 7, perturb=0.1, seed=1, fp32=False)  # four blocks per element
    x = torch.from_numpy(inputs.random_vector(m.n_global, seed=2)).cuda()
    y = {}
    for v in (3, 67):
        hb.hb_set_kernel_variant(m.handle, hb.HB_F64, v)
        y[v] = m.apply_A(x, lam=0.1)
    assert torch.equal(y[3], y[67])
    m.close()
