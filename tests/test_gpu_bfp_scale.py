"""The space-time product with coefficients near the ends of FP64's range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,timevar", [(5, False), (63, False), (300, True), (1023, False)])
def test_coefficients_of_any_magnitude(m, timevar):
    """d+, d- times 2^1000: the products' J part is 2^1000 times the plain one's, every intermediate
    included, and the A part vanishes beside it.  With the A part from the difference of two plain
    products (d and 2 d) each side carries a few roundings of its row's largest entry: 64 units."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDEProblem
    s, dev = 16, "cuda"
    x = torch.arange(1, m + 1, dtype=torch.float64, device=dev) / (m + 1)
    u0, f = 1.0 + x, torch.zeros((s + 1) * m, dtype=torch.float64, device=dev)
    z = torch.as_tensor(np.random.default_rng(m).standard_normal(m * s), device=dev)

    def products(scale):
        dp, dm = (1.0 + x) * scale, (2.0 - x) * scale
        more = {}
        if timevar:
            t = 1.0 + torch.linspace(0, 1, s + 1, dtype=torch.float64, device=dev)[:, None]
            more = dict(dplus_t=(t * dp).contiguous(), dminus_t=(t * dm).contiguous())
        with FDEProblem(m=m, s=s, alpha=1.6, xL=0.0, xR=1.0, t0=0.0, T=1.0, dplus=dp, dminus=dm, u0=u0, f=f,
                        family="GBDF", mu=3, **more) as p:
            p.assemble()
            return p.matvec(z).reshape(s, m), p.rhs().clone().reshape(s, m)

    one, two, big = products(1.0), products(2.0), products(2.0 ** 1000)
    for a, b, c in zip(one, two, big):
        assert torch.isfinite(c).all()
        ref, got = b - a, c * 2.0 ** -1000
        size = torch.maximum(a.abs(), b.abs()).amax(dim=1, keepdim=True)
        assert ((got - ref).abs() <= 64 * 2.0 ** -53 * size).all()
