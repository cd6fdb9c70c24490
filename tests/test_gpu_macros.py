"""rho^N and u of cgevap_get_macros are quotients rounded once: bit for bit torch's division of the same
numerators by the same density, so that a cell of one colour has rho^N = +-1."""
import pytest
import torch

from paper_2412_14859_gb300 import inputs
from paper_2412_14859_gb300.binding import Sim

pytestmark = pytest.mark.gpu

LATTICES = [(9, (1, 33, 65)), (19, (7, 9, 33))]


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("q,shape", LATTICES)
def test_phase_field_is_a_division(q, shape, storage):
    c = inputs.Case("m", q, shape, R0=3.0, noise=1e-6, rho_r_in=4.9, tau_b=0.8)
    sim = Sim.from_case(c, storage)
    g = torch.Generator().manual_seed(5)
    rn0 = (torch.rand(shape, generator=g, dtype=torch.float64) * 2 - 1)
    rn0.view(-1)[0::3] = 1.0
    rn0.view(-1)[1::3] = -1.0
    sim.init_equilibrium(rn0.cuda())
    m = sim.macros()
    rn = m["rhoN"].cpu()
    assert torch.equal(rn, ((m["rho_r"] - m["rho_b"]) / (m["rho_r"] + m["rho_b"])).cpu())
    assert (rn.view(-1)[0::3] == 1.0).all() and (rn.view(-1)[1::3] == -1.0).all()


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("q,shape", LATTICES)
def test_velocity_is_a_division(q, shape, storage):
    """Populations at rest and along +x and the march axis only: j is one of them."""
    c = inputs.Case("m", q, shape, R0=3.0)
    sim = Sim.from_case(c, storage)
    g = torch.Generator().manual_seed(6)
    f = torch.zeros((2, q) + shape, dtype=torch.float64)
    x, m_dir, m_axis = 1, 3 if q == 9 else 5, 1 if q == 9 else 2
    for i in (0, x, m_dir):
        f[0, i] = (torch.rand(shape, generator=g) + 0.1).double()  # FP32 values
    sim.set_populations(f.cuda())
    u = sim.macros()["u"].cpu()
    rho = f[0, 0] + f[0, x] + f[0, m_dir]
    assert torch.equal(u[0], f[0, x] / rho)
    assert torch.equal(u[m_axis], f[0, m_dir] / rho)
