"""The split of a 2D grid into regions that take several steps per launch
(csrc/step2d_tile.cu), at the edges that tests/test_gpu_tile2d.py does not
reach.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    import __graft_entry__ as ge
    ge.build()
    from paper_2509_15744_gb300 import wave
    return wave


def _final_levels(W, shape, physics, order, bc, nt):
    """(levels and launches of one forward call, levels of single steps)."""
    rng = np.random.default_rng(11)
    if physics == "velocity":
        p, h, vmax = rng.uniform(1500, 3000, shape), 10.0, 3000.0
    else:
        p, h, vmax = rng.uniform(0.1, 1.0, shape), 2e-3, 509.8366
    p = torch.from_numpy(p.astype(np.float32)).cuda()
    m = W.Model(p, h, O.cfl_dt(h, vmax, 2, order, 0.5), order, physics, bc)
    init = torch.from_numpy(rng.standard_normal((2,) + shape).astype(np.float32)).cuda()
    shot = W.Shot(0, torch.zeros(nt + 1, device="cuda"), torch.zeros(0, dtype=torch.int64, device="cuda"))
    before = W.launch_count()
    _, final = m.forward([shot], init=init, return_final=True)
    launches = W.launch_count() - before
    a, b = (torch.zeros(m.pitched_shape(), device="cuda") for _ in range(2))
    a[:, :shape[1]], b[:, :shape[1]] = init[0], init[1]
    for _ in range(nt):
        m.step([b], [a])
        a, b = b, a
    torch.cuda.synchronize()
    return final, launches, torch.stack([a[:, :shape[1]], b[:, :shape[1]]])


# few rows: three or four CTAs per SM, which overlapping launches share; each
# takes all (density) of the SM's tensor memory
@pytest.mark.parametrize("shape", [(16, 12000), (20, 6000), (23, 5000)])
def test_thin_density_grids_have_the_bits_of_single_steps(W, shape):
    final, launches, ref = _final_levels(W, shape, "density", 2, "neumann", 61)
    assert launches < 61   # several steps per launch
    assert torch.equal(final, ref)
