"""A x alone may start while the kernel before it drains: chains with
read-after-write and write-after-read between the calls, two streams side by
side, and capture in a caller's CUDA graph (where it may not) give the values of
the same calls one at a time."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2202_12477_gb300 import hb, inputs  # noqa: E402

# clusters of four and two blocks per element, one block, base shape
MESHES = [((3, 3, 3), 7, hb.HB_F64), ((4, 4, 4), 7, hb.HB_F64), ((5, 5, 5), 3, hb.HB_F64), ((12, 11, 12), 3, hb.HB_F64),
          ((3, 3, 2), 11, hb.HB_F64X), ((4, 4, 4), 5, hb.HB_F32)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.lib()


def _setup(dims, N, prec, seed):
    m = hb.Mesh(*dims, N, perturb=0.1, seed=seed, fp32=prec == hb.HB_F32)
    dt = torch.float32 if prec == hb.HB_F32 else torch.float64
    return m, torch.from_numpy(inputs.random_vector(m.n_global, seed=seed + 1)).to(dt).cuda()


def _chain(m, prec, x, steps, sync):
    """x <- A (A x) scaled, each buffer read by one call and overwritten by the next."""
    x = x.clone()
    y, z, seen = torch.empty_like(x), torch.empty_like(x), []
    for _ in range(steps):
        for a, b in ((x, y), (y, z), (z, x)):
            m.apply_A(a, b, lam=0.3, prec=prec)
            if sync:
                torch.cuda.synchronize()
        seen.append(y.clone())
        x.mul_(1e-6)
        if sync:
            torch.cuda.synchronize()
    return seen + [x]


@pytest.mark.parametrize("dims,N,prec", MESHES)
def test_chain_equals_one_at_a_time(dims, N, prec):
    m, x = _setup(dims, N, prec, 3)
    ref = _chain(m, prec, x, 12, True)
    for _ in range(5):
        got = _chain(m, prec, x, 12, False)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(ref, got))
    m.close()


@pytest.mark.parametrize("dims,N,prec", MESHES[:2])
def test_two_streams(dims, N, prec):
    sets = [_setup(dims, N, prec, seed) for seed in (3, 4)]
    refs = [_chain(m, prec, x, 12, True) for m, x in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    for _ in range(5):
        got = []
        torch.cuda.synchronize()
        for (m, x), s in zip(sets, streams):
            with torch.cuda.stream(s):
                got.append(_chain(m, prec, x, 12, False))
        torch.cuda.synchronize()
        for ref, g in zip(refs, got):
            assert all(torch.equal(a, b) for a, b in zip(ref, g))
    for m, _ in sets:
        m.close()


@pytest.mark.parametrize("dims,N,prec", MESHES)
def test_captured_in_a_graph(dims, N, prec):
    m, x = _setup(dims, N, prec, 5)
    y, z = torch.empty_like(x), torch.empty_like(x)
    m.apply_A(x, y, lam=0.3, prec=prec)  # first launches set attributes
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        m.apply_A(x, y, lam=0.3, prec=prec)
        m.apply_A(y, z, lam=0.3, prec=prec)
    for k in range(3):
        x.mul_(-0.5)
        g.replay()
        got = (y.clone(), z.clone())
        m.apply_A(x, y, lam=0.3, prec=prec)
        torch.cuda.synchronize()
        m.apply_A(y, z, lam=0.3, prec=prec)
        assert torch.equal(got[0], y) and torch.equal(got[1], z)
    m.close()
