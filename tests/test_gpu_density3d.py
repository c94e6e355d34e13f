"""The 3D density step that computes each face weight once (csrc/
step_density.cu, FP32): steps and increments against the oracle at the edges of
its split: one row tile more or less, a strip end inside a quad, a z-block of
one plane, the smallest grid.  (Two fields in one launch: the symmetric-mode
tests.)

Tolerances: a step is a few FP32 operations on values of order one: 1e-5 of
the largest value, the bar of the other one-step tests; increments 1e-5
relative L2.
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


def _setup(W, shape, bc, kahan, seed=3):
    rng = np.random.default_rng(seed)
    gamma = rng.uniform(0.1, 1.0, shape).astype(np.float32)
    dt = O.cfl_dt(2e-3, 509.8366, 3, 2, 0.5)
    m = W.Model(torch.from_numpy(gamma).cuda(), 2e-3, dt, 2, "density", bc, kahan=kahan)

    def pitched(a):
        out = np.zeros(shape[:-1] + (m.pitch,), np.float32)
        out[..., :shape[-1]] = a
        return torch.from_numpy(out).cuda()
    return rng, gamma, dt, m, pitched


@pytest.mark.parametrize("shape", [(3, 3, 3), (9, 8, 128), (8, 9, 129), (17, 7, 130), (4, 21, 259)])
@pytest.mark.parametrize("bc,kahan", [("dirichlet", False), ("neumann", True)])
def test_step_and_increment_match_the_oracle(W, shape, bc, kahan):
    rng, gamma, dt, m, pitched = _setup(W, shape, bc, kahan)
    cur, prev = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    med = O.Medium("density", gamma.astype(np.float64), 2e-3, dt, 2, bc)
    ref = med.step(prev.astype(np.float64), cur.astype(np.float64), np.zeros(shape))
    inc = -dt * (med.kernel_half_level(ref - cur, ref - cur) + med.kernel_level(cur.astype(np.float64), cur))
    for zb in (1, 8):
        m.set_block(zb)
        p = pitched(prev)
        acc, comp = (torch.zeros(m.pitched_shape(), device="cuda") for _ in range(2))
        m.step([pitched(cur)], [p], acc=acc, comp=comp if kahan else None)
        torch.cuda.synchronize()
        got = p.cpu().numpy()
        assert np.abs(got[..., :shape[-1]] - ref).max() < 1e-5 * np.abs(ref).max()
        a = acc.cpu().numpy()
        assert np.linalg.norm(a[..., :shape[-1]] - inc) < 1e-5 * np.linalg.norm(inc)
        assert not got[..., shape[-1]:].any() and not a[..., shape[-1]:].any()   # padding stays zero
