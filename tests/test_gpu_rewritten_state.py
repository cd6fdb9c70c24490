"""Buffers rewritten while a kernel that reads them runs: many ensemble steps in one launch (buffer c
is read in a step, written in the next and read again) against one step per launch, bit for bit, on
lattices small enough for an SM to keep lines of a buffer from one step to the next."""
import pytest
import torch

from paper_2412_14859_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f32x", "f64", "mixed"])
def test_many_steps_in_one_launch(storage):
    from paper_2412_14859_gb300.binding import Ensemble
    cases = [inputs.Case("a", 9, (1, 20, 31), R0=6.0, noise=1e-3, phi=3e-4),
             inputs.Case("b", 9, (1, 32, 16), R0=5.0, noise=1e-3, phi=1e-4, rho_r_in=2.0, tau_b=0.8),
             inputs.Case("c", 19, (6, 5, 33), R0=2.5, noise=1e-3, phi=3e-4),
             inputs.Case("d", 19, (8, 8, 8), R0=3.0, noise=1e-3, phi=1e-4, rho_r_in=2.0, tau_b=0.8)]
    st = ["f32", "f64"] * 2 if storage == "mixed" else storage
    ens = [Ensemble(cases, st) for _ in range(2)]
    for e in ens:
        for sim, c in zip(e.members, cases):
            sim.set_flux(c.phi)
            sim.init_equilibrium(torch.from_numpy(c.phase()).cuda(), torch.from_numpy(c.noise_array()).cuda())
    ens[0].step(41)
    for _ in range(41):
        ens[1].step(1)
    for a, b in zip(ens[0].members, ens[1].members):
        assert torch.equal(a.populations(), b.populations())
        assert torch.equal(a.mask(), b.mask())
        assert a.ledger() == b.ledger()
    for e in ens:
        e.status()
        e.close()
