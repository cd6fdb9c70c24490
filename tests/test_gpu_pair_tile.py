"""The pair storages' step at the edges of its tiles: one-plane, one-row and one-cell lattices,
tiles with one column over, and the two instantiations of the kernel -- the plain one (band rule,
scalar flux, no solids) and the general one -- which must give the same bits.

FP64 against the oracle at the parity tolerance of the other sizes, 1e-12 relative L-infinity."""
import numpy as np
import pytest
import torch

from paper_2412_14859_gb300 import inputs

from harness import gpu_sim, oracle_run, rel_linf

pytestmark = pytest.mark.gpu

SHAPES = [
    (9, (1, 1, 5)), (9, (1, 2, 128)), (9, (1, 9, 129)), (9, (1, 40, 127)),
    (19, (1, 4, 32)), (19, (2, 1, 33)), (19, (3, 5, 31)), (19, (9, 13, 65)), (19, (17, 8, 16)),
]
WALLS = [(1, 1, 1), (1, 1, 0), (0, 0, 1)]


def case(q, shape, periodic=(1, 1, 1), gamma=2.0):
    # S-bar a power of two: phi / S-bar and phi * (1 / S-bar) are the same bits
    return inputs.Case("edge", q, shape, periodic=periodic, R0=max(1.5, min(shape[1:]) / 3.0), noise=1e-3,
                       phi=3e-4, sbar=2.0, rho_r_in=gamma, tau_b=0.8)


@pytest.mark.parametrize("periodic", WALLS)
@pytest.mark.parametrize("q,shape", SHAPES)
def test_edge_shapes_fp64(q, shape, periodic):
    c = case(q, shape, periodic)
    run = oracle_run(c, 4)
    assert min(run.min_margin_history) > 1e-9
    sim = gpu_sim(c, "f64")
    sim.step(4)
    assert rel_linf(sim.populations().cpu().numpy(), run.f) <= 1e-12
    assert sim.ledger()["evaporated"] == pytest.approx(run.evaporated, rel=1e-12)


@pytest.mark.parametrize("storage", ["f64", "f32", "f32x"])
@pytest.mark.parametrize("q,shape", SHAPES)
def test_general_instantiation_gives_the_same_bits(q, shape, storage):
    c = case(q, shape)
    plain = gpu_sim(c, storage)
    field = gpu_sim(c, storage, phi_field=np.full(shape, c.phi))
    links = gpu_sim(c, storage)
    links.set_solid(torch.zeros(shape, dtype=torch.uint8, device="cuda"))
    for s in (plain, field, links):
        s.step(5)
    f = plain.populations()
    assert torch.equal(f, field.populations()) and torch.equal(f, links.populations())
    assert torch.equal(plain.mask(), field.mask()) and torch.equal(plain.mask(), links.mask())
    assert plain.ledger()["site_steps"] == field.ledger()["site_steps"] == links.ledger()["site_steps"]


@pytest.mark.parametrize("storage", ["f64", "f32", "f32x"])
@pytest.mark.parametrize("rule,periodic,extra", [
    (inputs.RULE_BAND, (1, 1, 1), ""), (inputs.RULE_GRADIENT, (1, 1, 1), ""), (inputs.RULE_BAND, (0, 0, 1), "field"),
    (inputs.RULE_GRADIENT, (1, 0, 1), "solid")])
@pytest.mark.parametrize("shape", [(1, 1, 9), (1, 7, 16), (1, 9, 33), (1, 70, 131)])
def test_patches_give_the_march_bits(shape, rule, periodic, extra, storage):
    """The D2Q9 step by patches against the marching one (chosen by a fixed chunk length)."""
    c = case(9, shape, periodic)
    c.site_rule, c.threshold = rule, 0.5 if rule == inputs.RULE_BAND else 0.1
    phi = c.phi * (1.0 + inputs.uniform_noise(shape, 0.5, seed=4)) if extra == "field" else None
    solid = (inputs.uniform_noise(shape, 1.0, seed=6) > 0.9).astype(np.uint8) if extra == "solid" else None
    a = gpu_sim(c, storage, phi_field=phi, solid=solid)
    b = gpu_sim(c, storage, phi_field=phi, solid=solid)
    b.tune(0, 0, min(3, shape[1]))
    a.step(6)
    b.step(6)
    assert torch.equal(a.populations(), b.populations())
    assert torch.equal(a.mask(), b.mask())
    la, lb = a.ledger(), b.ledger()
    assert la["site_steps"] == lb["site_steps"] and la["steps"] == lb["steps"] == 6
    # sums of the same terms in another order, over at most 6 x 9170 of them
    assert la["evaporated"] == pytest.approx(lb["evaporated"], rel=1e-11)


@pytest.mark.parametrize("q,shape", [(9, (1, 40, 127)), (19, (9, 13, 65))])
def test_steps_captured_in_a_graph(q, shape):
    """Steps launched ahead of their predecessor's end, captured and replayed."""
    c = case(q, shape)
    ref = gpu_sim(c, "f32")
    ref.step(10)
    sim = gpu_sim(c, "f32")
    sim.step(2)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sim.step(4)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(ref.populations(), sim.populations())
    assert ref.ledger()["site_steps"] == sim.ledger()["site_steps"]
