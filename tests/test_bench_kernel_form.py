"""The step kernel's name in the bench's records: the rare form where walls slide or a periodic lattice
is under eight columns wide, as the library chooses it."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from paper_2505_22256_gb300 import scenarios as S  # noqa: E402


def test_the_rare_form_is_named():
    sliding, plain = S.couette_channel(50, 40), S.cylinder_droplet(96)
    assert bench.rare_form([plain, sliding]) and not bench.rare_form([plain])
    still = S.couette_channel(9, 40)
    still.u_wall = (0.0, 0.0)
    assert not bench.rare_form([still])
    thin = S.couette_channel(7, 40)
    thin.u_wall = (0.0, 0.0)
    assert bench.rare_form([thin])
    thin.bc_x = "wall"
    assert not bench.rare_form([thin])
    info = {"wall_inline": 1, "block_threads": 64}
    assert bench.step_kernel_name("f32", info, True) == "k_step<float, float, 2, 1, 64>"
    assert bench.step_kernel_name("f32", info) == "k_step<float, float, 0, 1, 64>"
