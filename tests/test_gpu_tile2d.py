"""Several 2D steps per launch (csrc/step2d_tile.cu): regions of the grid that
overlap by the steps' halo.

The forward from given levels and no force must give the bits of the same
number of single steps (`Model.step`, the one-step kernel) at every edge of
the split: grids one region wide or high, one cell more than a region, last
regions at unaligned offsets, step counts that leave a remainder.  Gradients
with receivers in several regions, duplicated receivers and receivers outside
the grid are held to the oracle at the parity bars of the other tests (traces
1e-4, sensitivity 1e-3 at the same k).
"""
import numpy as np
import pytest
import torch

import oracle as O
from _gpu import gpu_model, gpu_shots
from _problems import make_problem, rel_l2

pytestmark = pytest.mark.gpu

SHAPES = [(16, 128), (17, 129), (64, 128), (65, 131), (130, 257), (203, 383), (19, 2501)]


@pytest.fixture(scope="module")
def W():
    import __graft_entry__ as ge
    ge.build()
    from paper_2509_15744_gb300 import wave
    return wave


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("physics,order,bc,nt", [
    ("velocity", 2, "dirichlet", 61), ("velocity", 4, "neumann", 33), ("velocity", 6, "dirichlet", 23),
    ("velocity", 8, "neumann", 19), ("velocity", 8, "dirichlet", 1), ("density", 2, "dirichlet", 41),
    ("density", 2, "neumann", 40)])
def test_forward_has_the_bits_of_single_steps(W, shape, physics, order, bc, nt):
    rng = np.random.default_rng(7)
    if physics == "velocity":
        p, h, vmax = rng.uniform(1500, 3000, shape), 10.0, 3000.0
    else:
        p, h, vmax = rng.uniform(0.1, 1.0, shape), 2e-3, 509.8366
    p = torch.from_numpy(p.astype(np.float32)).cuda()
    m = W.Model(p, h, O.cfl_dt(h, vmax, 2, order, 0.5), order, physics, bc)
    init = torch.from_numpy(rng.standard_normal((2,) + shape).astype(np.float32)).cuda()
    none = torch.zeros(0, dtype=torch.int64, device="cuda")
    shot = W.Shot(0, torch.zeros(nt + 1, device="cuda"), none)
    _, final = m.forward([shot], init=init, return_final=True)
    a, b = (torch.zeros(m.pitched_shape(), device="cuda") for _ in range(2))
    a[:, :shape[1]], b[:, :shape[1]] = init[0], init[1]
    for _ in range(nt):
        m.step([b], [a])
        a, b = b, a
    torch.cuda.synchronize()
    assert torch.equal(final[0], a[:, :shape[1]])
    assert torch.equal(final[1], b[:, :shape[1]])


@pytest.mark.parametrize("shape,order,bc,kahan,objective", [
    ((65, 131), 2, "neumann", False, "l2"), ((130, 257), 4, "dirichlet", True, "l2"),
    ((77, 150), 8, "dirichlet", False, "patch"), ((40, 300), 6, "neumann", True, "patch")])
def test_gradient_matches_the_oracle(W, shape, order, bc, kahan, objective):
    ny, nx = shape
    if objective == "patch":   # dense: more entries than threads in the regions that hold it
        yy, xx = np.meshgrid(np.arange(8, ny - 8), np.arange(20, 100), indexing="ij")
        kw = dict(patch=(yy * nx + xx).ravel(), src=(ny // 2) * nx + 12)
    else:                      # on the edges, twice in one cell, on the source
        rec = np.unique(np.concatenate([np.arange(0, nx, 3), (ny - 1) * nx + np.arange(0, nx, 3),
                                        np.arange(0, ny * nx, nx), np.arange(nx - 1, ny * nx, nx)]))
        kw = dict(rec=np.concatenate([rec, rec[:5], [2 * nx + 30]]), src=2 * nx + 30)
    prob = make_problem(shape, order, bc, nt=60, seed=5, objective=objective, **kw)
    m = gpu_model(W, prob, kahan=kahan)
    g, c, k = m.gradient(gpu_shots(W, prob), objective=objective)
    ref = O.superposition_gradient(prob.medium(), prob.oracle_shots(), prob.nt[0], float(k.item()))
    assert rel_l2(g.cpu().numpy(), ref["K_tilde"]) < 1e-3
    assert abs(float(c.item()) - ref["C"]) < 1e-5 * abs(ref["C"])


@pytest.mark.parametrize("shape,physics,order,bc,mode,kahan", [
    ((65, 131), "velocity", 2, "neumann", "symmetric", False),
    ((70, 257), "velocity", 8, "dirichlet", "symmetric", True),
    ((66, 129), "velocity", 4, "neumann", "reverse", False),
    ((20, 300), "velocity", 6, "dirichlet", "reverse", True)])
def test_two_field_modes_match_the_exact_gradient(W, shape, physics, order, bc, mode, kahan):
    prob = make_problem(shape, order, bc, physics, nt=50, nrec=60, seed=6, nshots=2)
    m = gpu_model(W, prob, kahan=kahan)
    g, c, _ = m.gradient(gpu_shots(W, prob), mode=mode)
    cref, ref, _ = O.exact_gradient(prob.medium(), prob.oracle_shots(), prob.nt[0])
    assert rel_l2(g.cpu().numpy(), ref) < 1e-3
    assert abs(float(c.item()) - cref) < 1e-5 * abs(cref)


def test_density_symmetric_mode_over_several_regions(W):
    # the problem of the one-region test of this mode, on a taller grid
    prob = make_problem((130, 150), physics="density", bc="dirichlet", nt=200, nrec=40, seed=62)
    m = gpu_model(W, prob, kahan=True)
    g, c, _ = m.gradient(gpu_shots(W, prob), mode="symmetric")
    cref, ref, _ = O.exact_gradient(prob.medium(), prob.oracle_shots(), prob.nt[0])
    assert rel_l2(g.cpu().numpy(), ref) < 1e-3
    assert abs(float(c.item()) - cref) < 1e-5 * abs(cref)


def test_receivers_outside_the_grid_record_zero(W):
    prob = make_problem((66, 140), 4, "dirichlet", nt=30, nrec=20, seed=9)
    m = gpu_model(W, prob)
    s = gpu_shots(W, prob)[0]
    far = torch.tensor([66 * 140, 10 ** 12, -1], dtype=torch.int64, device="cuda")
    with_far = W.Shot(s.src, s.wavelet, torch.cat([far[:1], s.rec, far[1:]]))
    ref = m.forward([W.Shot(s.src, s.wavelet, s.rec)])[0]
    got = m.forward([with_far])[0]
    torch.cuda.synchronize()
    assert torch.equal(got[1:-2], ref)
    assert not got[0].any() and not got[-2:].any()


@pytest.mark.parametrize("physics,mode", [("velocity", "superposition"), ("velocity", "reverse"),
                                          ("density", "symmetric")])
def test_overlapping_launches_captured_in_a_cuda_graph(W, physics, mode):
    # the launches of a pass start while the one before ends; captured, replayed
    # and on another stream they give the bits of the eager call
    prob = make_problem((70, 150), 2, "neumann", physics, nt=90, nrec=30, seed=11)
    m, shots = gpu_model(W, prob), gpu_shots(W, prob)
    eager, c, _ = m.gradient(shots, mode=mode, k=1.0)
    out = torch.empty_like(eager)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _, cg, _ = m.gradient(shots, mode=mode, k=1.0, out=out)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, eager) and float(cg.item()) == float(c.item())
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        again, c2, _ = m.gradient(shots, mode=mode, k=1.0)
    side.synchronize()
    assert torch.equal(again, eager) and float(c2.item()) == float(c.item())
