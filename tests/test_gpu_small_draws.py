"""The constant-hazard draws of the one-warp kernel at the ends of their ranges: hazards at which every gap is zero, at
which hardly any slot ends, several blocks of draws per worker, gap tables of few slots; and arrivals beyond 32 a
step.  Whole numbers against the checker: equality."""
import pytest

from paper_2605_06113_b200 import workload as wlm
from helpers import run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hazard", [0.0, 1e-7, 1e-3, 0.12, 0.5, 0.97, 1.0])
@pytest.mark.parametrize("G,B,W,lam", [(32, 64, 256, 20.0), (5, 8, 36, 3.0), (31, 56, 512, 55.0)])
def test_draws_at_extreme_hazards(hazard, G, B, W, lam):
    cfg = wlm.get_config("c3", G=G, B=B, W=W, init_active=B - B // 8, init_queue=W // 2, hazard=hazard,
                         arrival=("const", lam), S_greedy=-1)
    run_parity(cfg, 2, 24, threads=32, launch_steps=4, check_every=1)
