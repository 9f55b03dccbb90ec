"""Which meshes the fused CG takes: mode 2 whenever one block per element fits
on the GPU at once (5 x 152 elements at N = 1..3 and 6, 4 x 152 at N = 4, 5, 7, 8,
2 x 152 at N = 9, 10, 152 from N = 11 on), the default up to 300 of them, less few
and large elements."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def _fused_launches(dims, N, mode):
    m = hb.Mesh(*dims, N, perturb=0.1, seed=1, fp32=False)
    hb.lib().hb_set_cg_fused(m.handle, mode)
    b = m.rhs(kind=0, seed=2)
    hb.hb_profile_enable(True)
    try:
        hb.hb_profile_reset()
        x, res = m.cg(b, lam=0.3, max_it=5)
        count = hb.hb_profile_read("cg_fused")[1]
    finally:
        hb.hb_profile_enable(False)
    hb.lib().hb_set_cg_fused(m.handle, 1)
    y, _ = m.cg(b, lam=0.3, max_it=5)
    assert res.status == hb.HB_OK and float((x - y).norm()) <= 1e-12 * float(y.norm())
    m.close()
    return count


@pytest.mark.parametrize("N,dims", [(1, (20, 19, 2)), (2, (20, 19, 2)), (3, (20, 19, 2)), (4, (19, 16, 2)),
                                    (5, (19, 16, 2)), (6, (20, 19, 2)), (7, (19, 16, 2)), (8, (19, 16, 2)),
                                    (9, (19, 16, 1)), (10, (19, 16, 1)), (11, (19, 8, 1)), (15, (19, 8, 1))])
def test_mode_2_takes_every_mesh_that_fits(N, dims):
    assert _fused_launches(dims, N, 2) == 1
    assert _fused_launches((dims[0], dims[1], dims[2] + 3), N, 2) == 0


@pytest.mark.parametrize("N,dims,fused", [(5, (6, 6, 6), 1), (9, (6, 6, 6), 1), (10, (6, 6, 6), 1), (7, (7, 7, 6), 1),
                                          (7, (7, 7, 7), 0), (11, (6, 5, 5), 1), (11, (4, 4, 4), 0), (10, (4, 4, 4), 1),
                                          (10, (3, 3, 3), 0), (15, (5, 5, 5), 1), (15, (2, 2, 2), 0)])
def test_default_range(N, dims, fused):
    assert _fused_launches(dims, N, 0) == fused
