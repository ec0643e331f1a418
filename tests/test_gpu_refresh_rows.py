"""Refreshes of c_hat from classifier rows of every width that is loaded as a whole (8, 4, 2 probabilities, or one by one) and
of every horizon group, with lists of due requests that fill their warp's part, run over a round of rows or
stay empty.  Whole numbers and fp32 c_hat against the checker: the tolerance is equality."""
import pytest

from paper_2605_06113_b200 import workload as wlm
from helpers import run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [0, 32, 256])
@pytest.mark.parametrize("G,B,H,delta_T", [
    (3, 8, 1, 1), (5, 24, 2, 1), (21, 40, 6, 3), (7, 40, 7, 1), (9, 64, 4, 2), (16, 64, 8, 1), (40, 64, 8, 4), (11, 72, 9, 2),
    (6, 64, 11, 5), (6, 64, 12, 1), (5, 40, 16, 1), (40, 24, 18, 9), (3, 40, 20, 1), (2, 256, 27, 13),
])
def test_rows_of_every_width(G, B, H, delta_T, threads):
    for gate, active in ((0.02, B), (0.5, B - B // 4)):
        cfg = wlm.get_config("c2", G=G, B=B, W=64, H=H, init_active=active, init_queue=60, hazard=0.03, term_mode=1, gate=gate,
                             delta_T=delta_T, score_mode=-1, S_greedy=-1, arrival=("const", 3.0))
        run_parity(cfg, 3, 6, threads=threads, launch_steps=2, check_every=1)
