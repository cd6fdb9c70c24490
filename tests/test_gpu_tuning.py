"""cgevap_get_tuning's values, given back to cgevap_tune, keep the plan: chunks, D2Q9 patches and the even
shares of FP64.  The reverse sweep refuses a plan other than its forward run's, which shows a change."""
import pytest
import torch

from harness import gpu_sim
from paper_2412_14859_gb300 import inputs

pytestmark = pytest.mark.gpu

# (lattice, shape, storage, the plan is chunks); 640 FP64 tiles of 9 planes go to even shares
PLANS = [(9, (1, 24, 33), "f32", False), (9, (1, 24, 33), "f64", False), (19, (6, 9, 33), "f32", True),
         (19, (6, 9, 33), "f64", True), (19, (9, 157, 509), "f64", False)]


@pytest.mark.parametrize("q,shape,storage,chunks", PLANS)
def test_round_trip_keeps_the_plan(q, shape, storage, chunks):
    sim = gpu_sim(inputs.Case("t", q, shape, R0=3.0, phi=1e-4), storage)
    t = sim.tuning()
    assert (t["planes_per_chunk"] > 0) == chunks
    sim.adjoint_forward(2)
    sim.tune(**t)
    assert sim.tuning() == t
    sim.adjoint_backward(torch.ones(3, dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("q,shape,storage", [p[:3] for p in PLANS])
def test_a_fixed_length_is_reported(q, shape, storage):
    sim = gpu_sim(inputs.Case("t", q, shape, R0=3.0, phi=1e-4), storage)
    sim.tune(0, 0, 2)
    assert sim.tuning() == {"family": 0, "variant": 0, "planes_per_chunk": 2}
    sim.tune(0, 0, 10 ** 6)
    assert sim.tuning()["planes_per_chunk"] == (shape[1] if q == 9 else shape[0])
