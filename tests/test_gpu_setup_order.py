"""First calls right after a set-up, on a side stream that does not wait for
the default one: tables, item lists and zeroed buffers that the set-up
uploads or fills have to be in place.  The first result equals a repeated one
bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


@pytest.mark.parametrize("L,nlon,prec", [(31, 96, "fp64"), (100, 324, "fp64"), (53, 162, "fp32"), (255, 768, "fp32"),
                                         (127, 384, "bf16x3"), (255, 768, "bf16x3")])
def test_first_rhs_on_a_side_stream(L, nlon, prec):
    from paper_1009_3308_gb300 import Plan
    a = _dev(coefficients(L, 7, 3.0 / L))
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        plan = Plan(L, nlon // 2, nlon, 1e-3, 1.0, precision=prec)
        first = plan.rhs(a)
        again = plan.rhs(a)
        J, g = plan.objective(a, torch.zeros_like(a), 0.5, 1.0)
        J2, g2 = plan.objective(a, torch.zeros_like(a), 0.5, 1.0)
    torch.cuda.synchronize()
    assert torch.equal(first, again)
    assert J == J2 and torch.equal(g, g2)


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
def test_first_ensemble_calls_on_a_side_stream(prec):
    from paper_1009_3308_gb300 import Ensemble
    Ls = [63, 127, 63]
    al = [_dev(coefficients(L, 20 + i, 0.05)) for i, L in enumerate(Ls)]
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        ens = Ensemble(Ls, [1e-3, 1e-4, 1e-5], 1.0, precision=prec)
        for i, a in enumerate(al):
            ens.set_alpha(i, a)
        ens.rhs()
        first = [ens.get(i, "F") for i in range(3)]
        assert all(torch.equal(ens.get(i), a) for i, a in enumerate(al))
        ens.rhs()
        again = [ens.get(i, "F") for i in range(3)]
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(first, again))
