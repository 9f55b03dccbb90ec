"""The variant of A x alone: by the size rule on an untouched mesh, what was set
where a caller set one, and what was measured after tuning; an excluded lattice
gather stays excluded on meshes large enough for the rule."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import autotune, hb, inputs  # noqa: E402

GRID = hb.HB_VARIANT_GRID


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


@pytest.mark.parametrize("dims,N,prec", [((20, 20, 19), 15, hb.HB_F32), ((40, 39, 41), 7, hb.HB_F64X),
                                         ((80, 81, 80), 3, hb.HB_F64), ((4, 4, 4), 7, hb.HB_F64)])
def test_apply_variant(dims, N, prec, tmp_path):
    def mesh():
        return hb.Mesh(*dims, N, perturb=0.1, seed=2, fp32=prec == hb.HB_F32)
    m = mesh()
    large = m.n_local >= 30_000_000
    x = torch.from_numpy(inputs.random_vector(m.n_global, seed=6)).to(torch.float32 if prec == hb.HB_F32 else
                                                                      torch.float64).cuda()
    default = m.apply_A(x, lam=0.4, prec=prec)
    assert hb.hb_get_kernel_variant(m.handle, prec) == 3
    assert hb.hb_get_apply_variant(m.handle, prec) == (3 | GRID if large else 3)
    hb.hb_set_kernel_variant(m.handle, prec, 3)  # a caller's choice is what runs
    assert hb.hb_get_apply_variant(m.handle, prec) == 3
    assert torch.equal(m.apply_A(x, lam=0.4, prec=prec), default)
    hb.hb_set_apply_variant(m.handle, prec, 67)
    assert hb.hb_get_kernel_variant(m.handle, prec) == 3 and hb.hb_get_apply_variant(m.handle, prec) == 67
    assert torch.equal(m.apply_A(x, lam=0.4, prec=prec), default)
    with pytest.raises(hb.HBError):
        hb.hb_set_apply_variant(m.handle, prec, 6)
    path = str(tmp_path / "c.json")
    for exclude in (GRID, 0):
        v = autotune.tune_mesh(m, precs=(prec,), path=path, reps=2, exclude=exclude)[prec]
        ax = hb.hb_get_apply_variant(m.handle, prec)
        assert v == hb.hb_get_kernel_variant(m.handle, prec) and not (ax & exclude) and not (v & exclude)
        assert ax == v or (large and ax == (v & ~hb.HB_VARIANT_CSR) | GRID)
        m2 = mesh()  # from the cache
        assert autotune.tune_mesh(m2, precs=(prec,), path=path, exclude=exclude)[prec] == v
        assert hb.hb_get_apply_variant(m2.handle, prec) == ax
        m2.close()
    m.close()
