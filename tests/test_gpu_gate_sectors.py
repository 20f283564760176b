"""Gates whose controls or phases leave half sectors, in a state beyond the L2 and
in a small one: the same as amplitude by amplitude."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,n", [("c64", 8), ("c64", 24), ("c64", 25), ("c128", 8), ("c128", 24)])
@pytest.mark.parametrize("target,controls", [(1, ()), (0, (1,)), (1, (2,)), (6, (1,)), (6, (2, 3)), (6, (1, 2, 7)), (2, (5,))])
def test_phases_and_flips(svlib, dt, n, target, controls):
    """A product of two numbers of relative error eps: 4 eps of each amplitude; a
    flip moves amplitudes exactly."""
    s = svlib.StateVector(n, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    s.amps.normal_(generator=g)
    amps = torch.view_as_complex(s.amps.view(-1, 2))
    psi = amps.clone()
    x = torch.arange(1 << n, device="cuda")
    on = torch.ones_like(x, dtype=torch.bool)
    for c in controls:
        on &= (x >> c) & 1 == 1
    phase = complex(np.exp(0.7j))
    s.apply_gate(np.diag([1, phase]), [target], list(controls))
    want = torch.where(on & ((x >> target) & 1 == 1), psi.to(torch.complex128) * phase, psi.to(torch.complex128))
    eps = 2.0 ** -23 if dt == "c64" else 2.0 ** -52
    assert ((amps.to(torch.complex128) - want).abs() <= 4 * eps * want.abs()).all()
    amps.copy_(psi)
    s.apply_gate(np.array([[0, 1], [1, 0]], dtype=complex), [target], list(controls))
    assert torch.equal(amps, torch.where(on, psi[x ^ (1 << target)], psi))
    s.close()
