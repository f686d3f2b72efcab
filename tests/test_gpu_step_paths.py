"""Forward-step kernels at the sizes where their dispatch or tiling changes, against the oracle."""
import numpy as np
import pytest

from paper_2605_27004_gb300 import inputs
from gpu_util import gpu_run, oracle_run, perm_lib_to_oracle, rand_theta

pytestmark = pytest.mark.gpu


# FP64 steps run 64-thread blocks (rows of 1, 31, 32, 33, 65 cells: remainders of a warp and of a
# block; 70,001 rows: more than 64-thread blocks can cover in grid.y). Per step the collision
# rounds each population to about 10 * 2^-53 of f <= 0.5, so 20 steps stay below 1e-13.
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("q,dims", [(9, (1, 7, 1)), (9, (31, 9, 1)), (9, (65, 4, 1)), (9, (2, 70001, 1)),
                                    (19, (33, 3, 5)), (19, (32, 4, 2)), (27, (65, 2, 3))])
def test_fp64_step_block_edges(q, dims, scheme):
    d, N = (2 if q == 9 else 3), int(np.prod(dims))
    Th = rand_theta(5, d)
    rho0, u0 = inputs.noise_field(N, d, 0.05, 6, rho_amp=0.02)
    g = gpu_run(q, dims, 0.8, Th, rho0, u0, 20, storage="fp64", scheme=scheme)
    o = oracle_run(q, dims, 0.8, Th, rho0, u0, 20)
    assert np.abs(g["f"] - o["f"][:, perm_lib_to_oracle(q)].T).max() < 1e-13
