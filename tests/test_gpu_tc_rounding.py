"""The tensor-core FP64 element kernel rounds its digit sums to nearest: the
gradient of a constant is zero. D's integers sum to at most n 2^-9 units a row
(each is rounded to 2^-8), times 2^54 for the constant 1: below half of the 2^50
that a sum is rounded to. (Cut off instead of rounded, every negative sum
becomes -2^50, and A 1 is not zero.)"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


@pytest.mark.parametrize("N", hb.TC_DEGREES)
@pytest.mark.parametrize("variant", hb.VARIANTS_TC)
def test_constant_has_no_gradient(N, variant):
    m = hb.Mesh(3, 2, 3, N, perturb=0.1, seed=3, faces=0, fp32=False)
    hb.hb_set_kernel_variant(m.handle, hb.HB_F64, variant)
    for c in (1.0, -1.0, 2.0 ** -40):
        x = torch.full((m.n_global,), c, dtype=torch.float64, device="cuda")
        assert torch.count_nonzero(m.apply_A(x, lam=0.0)).item() == 0
    m.close()
