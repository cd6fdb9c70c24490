"""FP64 steps whose CTAs take even shares of all tiles' planes, against the same lattice marched in
chunks: shares longer than a tile's planes (three and more pieces) and shorter ones, that end inside
ragged tiles, with walls, solids and flux fields whose loads cross from one tile to the next.

The two plans start their marches at other planes, where the last bit of rho^N at a site may differ, so
populations agree to the FP64 parity tolerance (1e-12 relative) and site bytes and counts exactly."""
import numpy as np
import pytest
import torch

from harness import gpu_sim
from paper_2412_14859_gb300 import inputs

pytestmark = pytest.mark.gpu

# share of planes per CTA on 152 SMs with two CTAs each: 19, 15, 19 and 23
SHAPES = [(9, 157, 509), (13, 140, 300), (17, 150, 257), (30, 150, 190)]
KINDS = [("band", (1, 1, 1), ""), ("band", (1, 1, 0), "field"), ("gradient", (0, 1, 1), "solid"),
         ("gradient", (0, 0, 0), "solid+field")]


@pytest.mark.parametrize("rule,periodic,extra", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
def test_shares_equal_chunks(shape, rule, periodic, extra):
    band = rule == "band"
    c = inputs.Case("shares", 19, shape, periodic=periodic, R0=0.4 * min(shape[1:]), noise=1e-6, phi=3e-4, sbar=2.0,
                    rho_r_in=2.0, tau_b=0.8, site_rule=inputs.RULE_BAND if band else inputs.RULE_GRADIENT,
                    threshold=0.5 if band else 0.1)
    phi = c.phi * (1.0 + inputs.uniform_noise(shape, 0.5, seed=4)) if "field" in extra else None
    solid = (inputs.uniform_noise(shape, 1.0, seed=6) > 0.9).astype(np.uint8) if "solid" in extra else None
    shares = gpu_sim(c, "f64", phi_field=phi, solid=solid)
    chunks = gpu_sim(c, "f64", phi_field=phi, solid=solid)
    assert shares.tuning()["planes_per_chunk"] == 0
    chunks.tune(0, 0, 5)
    shares.step(3)
    chunks.step(3)
    a, b = shares.populations(), chunks.populations()
    assert float((a - b).abs().max() / b.abs().max()) <= 1e-12
    assert torch.equal(shares.mask(), chunks.mask())
    la, lb = shares.ledger(), chunks.ledger()
    assert la["site_steps"] == lb["site_steps"] > 0 and la["steps"] == 3
    assert la["evaporated"] == pytest.approx(lb["evaporated"], rel=1e-12)
