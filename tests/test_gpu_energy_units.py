"""A step does not depend on the unit of energy: H scaled by s and the step size by 1 / s give the same state.

With s a power of two every product and sum of the step is scaled exactly, so the states agree to the rounding of the few places
where a constant enters (1e-12 is asserted, the bound of the other step tests).
"""
import types

import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


def _run(w, s, scheme):
    b = w.bonds
    bonds = types.SimpleNamespace(site_i=b.site_i, site_j=b.site_j, jxy=np.asarray(b.jxy) * s, jz=np.asarray(b.jz) * s)
    L = Lrei(w.n, bonds, [x * s for x in w.B], w.kappa, "qll", "fp64", w.r)
    L.set_state(torch.from_numpy(w.V).cuda(), w.lam)
    L.step(0.01 / s, scheme, 5)
    V, lam, _ = L.get_state()
    return (V * torch.as_tensor(lam, device="cuda")) @ V.mH


@pytest.mark.parametrize("scheme", ["rk4", "ab3"])
@pytest.mark.parametrize("exponent", [-330, -40, 40, 330])
def test_step(exponent, scheme):
    w = li.workload(2, n=8, r=5)
    ref = _run(w, 1.0, scheme)
    assert float((_run(w, 2.0 ** exponent, scheme) - ref).abs().max()) < 1e-12
