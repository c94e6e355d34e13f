"""The split of a 2D grid into regions that take several steps per launch
(csrc/step2d_tile.cu), at the edges that tests/test_gpu_tile2d.py does not
reach.
"""
import numpy as np
import pytest
import torch

import oracle as O
from _gpu import gpu_model, gpu_shots
from _problems import make_problem

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


def _calls(W, prob, mode, **kw):
    """One forward and one gradient call through the C entry, each with the
    full and with the least workspace: {entry: [(outputs, launches, bytes)]}."""
    m, shots = gpu_model(W, prob, **kw), gpu_shots(W, prob)
    st, out = W._stream(), {"forward": [], "gradient": []}

    def run(call, nbytes):
        ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        before = W.launch_count()
        assert call(W._vp(ws.data_ptr()), nbytes) == 0
        launches = W.launch_count() - before
        assert call(W._vp(ws.data_ptr()), least.value - 1) == 3   # too small
        torch.cuda.synchronize()
        return launches
    o = W.GradOpts()
    o.objective, o.mode, o.k = W.OBJECTIVE[prob.objective], W.MODE[mode], 1.0
    o.patch_sign = 1.0
    for entry in out:
        full, least = W._sz(0), W._sz(0)
        for size in ("full", "least"):
            if entry == "forward":
                res = [torch.empty(s.nrec, s.nt + 1, device="cuda") for s in shots]
                arr = W._shot_descs(shots, res)
                assert W._fwd_ws(m._h, arr, len(shots), W.C.byref(full)) == 0
                assert W._fwd_min(m._h, arr, len(shots), W.C.byref(least)) == 0

                def call(p, n):
                    return W._forward(m._h, arr, len(shots), None, None, p, n, st)
            else:
                res = [torch.empty(prob.shape, device="cuda")]
                arr = W._shot_descs(shots)
                assert W._grad_ws(m._h, arr, len(shots), W.C.byref(o), W.C.byref(full)) == 0
                assert W._grad_min(m._h, arr, len(shots), W.C.byref(o), W.C.byref(least)) == 0

                def call(p, n):
                    return W._adjoint_sensitivity(m._h, arr, len(shots), W.C.byref(o), W._ptr(res[0]), None, None,
                                                  None, p, n, st)
            n = {"full": full, "least": least}[size].value
            out[entry].append((res, run(call, n), n))
    return out


# two rows or four per warp, one wave of regions or several, thin grids, order
# 6 with several steps per launch; sources and receivers in several regions
@pytest.mark.parametrize("shape,physics,order,bc,mode,kahan", [
    ((131, 257), "velocity", 2, "neumann", "superposition", False),
    ((600, 610), "velocity", 2, "neumann", "superposition", True),
    ((600, 610), "velocity", 8, "dirichlet", "superposition", False),
    ((700, 1500), "velocity", 8, "neumann", "superposition", True),
    ((700, 1501), "velocity", 4, "dirichlet", "reverse", False),
    ((700, 1500), "velocity", 2, "dirichlet", "symmetric", True),
    ((40, 131), "velocity", 6, "neumann", "superposition", True),
    ((90, 1400), "velocity", 6, "dirichlet", "symmetric", False),
    ((16, 3000), "velocity", 2, "neumann", "reverse", False),
    ((20, 6000), "density", 2, "dirichlet", "symmetric", True),
    ((800, 1300), "density", 2, "neumann", "superposition", True)])
def test_least_workspace_takes_single_steps_with_the_same_bits(W, shape, physics, order, bc, mode, kahan):
    ny, nx = shape
    rng = np.random.default_rng(13)
    src = [2 * nx + nx // 3, (ny // 2) * nx + 5]
    near = [s + dy * nx + dx for s in src for dy in range(-2, 7, 2) for dx in range(-5, 30, 3)]
    rec = np.setdiff1d(np.concatenate([near, rng.integers(0, ny * nx, 90)]), src)   # no cell takes two forces
    prob = make_problem(shape, order, bc, physics, nt=35, seed=13, nshots=2, src=src, rec=rec, objective="patch",
                        random_wavelet=True)
    prob.objective = "l2"
    prob.observed = [rng.standard_normal((rec.size, 36)).astype(np.float32) for _ in src]
    for entry, (full, least) in _calls(W, prob, mode, kahan=kahan).items():
        assert least[2] < full[2] and full[1] < least[1], entry   # less memory, more launches
        for a, b in zip(full[0], least[0]):
            assert torch.equal(a, b), entry
            assert a.any()


def test_model_falls_back_where_memory_is_short(W, monkeypatch):
    prob = make_problem((130, 257), 4, "dirichlet", nt=30, nrec=40, seed=14)
    shots = gpu_shots(W, prob)
    ref, rc, _ = gpu_model(W, prob).gradient(shots, k=1.0)
    m, real, asked = gpu_model(W, prob), W._workspace, []
    grid = 4 * 130 * m.pitch

    def short(nbytes, device):   # a device with room for three grids and a little
        asked.append(nbytes)
        if nbytes > 4 * grid:
            raise torch.OutOfMemoryError("out of memory")
        return real(nbytes, device)
    monkeypatch.setattr(W, "_workspace", short)
    for _ in range(2):
        g, c, _ = m.gradient(shots, k=1.0)
        assert torch.equal(g, ref) and float(c.item()) == float(rc.item())
    assert len(asked) == 2   # the full size once, the least once
    m2 = gpu_model(W, prob)

    def none(nbytes, device):
        raise torch.OutOfMemoryError("out of memory")
    monkeypatch.setattr(W, "_workspace", none)
    with pytest.raises(torch.OutOfMemoryError):
        m2.gradient(shots, k=1.0)


# Lists of the receivers per region are built once per call: a block of many
# receivers, whose regions share few counters, must not cost more than the
# steps it prepares.
def test_dense_receivers_do_not_slow_the_call_down(W):
    n, nt = 2048, 20
    m = W.Model(torch.full((n, n), 2500.0, device="cuda"), 10.0, O.cfl_dt(10.0, 2500.0, 2, 2, 0.5))
    shot = W.Shot(n // 2, torch.randn(nt + 1, device="cuda"), torch.arange(n * n // 4, 7 * n * n // 16, device="cuda"))
    traces = torch.empty(shot.nrec, nt + 1, device="cuda")
    arr, ms = W._shot_descs([shot], [traces]), {}
    for name, query in (("full", W._fwd_ws), ("least", W._fwd_min)):
        size = W._sz(0)
        assert query(m._h, arr, 1, W.C.byref(size)) == 0
        ws, times = torch.empty(size.value, dtype=torch.uint8, device="cuda"), []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            assert W._forward(m._h, arr, 1, None, None, W._ptr(ws), size.value, W._stream()) == 0
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms[name] = min(times)
    # several steps per launch against one: 0.43 and 0.56 ms; 1.6 ms with an atomic per receiver
    assert ms["full"] < 1.25 * ms["least"], ms


# calls that several steps per launch would slow down take one: they need no
# second pair of level grids
@pytest.mark.parametrize("shape,physics,order,mode,nt,dense,several", [
    ((251, 251), "velocity", 2, "superposition", 2, 0.0, False),
    ((251, 251), "velocity", 2, "superposition", 3, 0.0, True),
    ((251, 251), "density", 2, "superposition", 2, 0.0, False),
    ((251, 251), "density", 2, "symmetric", 2, 0.0, True),
    ((300, 400), "velocity", 4, "superposition", 20, 0.8, True),      # one wave of regions
    ((1000, 1300), "velocity", 2, "superposition", 20, 0.4, True),
    ((1000, 1300), "velocity", 2, "superposition", 20, 0.6, False),
    ((1000, 1300), "velocity", 8, "superposition", 20, 0.4, False),
    ((1000, 1300), "velocity", 8, "symmetric", 20, 0.2, False),
    ((1000, 1300), "velocity", 8, "superposition", 8, 0.1, False),
    ((1000, 1300), "density", 2, "symmetric", 20, 0.8, True),
    ((27, 300), "velocity", 6, "superposition", 30, 0.0, True),
    ((25, 300), "velocity", 6, "superposition", 30, 0.0, False)])
def test_route_of_short_records_and_dense_receivers(W, shape, physics, order, mode, nt, dense, several):
    n = shape[0] * shape[1]
    p = torch.full(shape, 2500.0 if physics == "velocity" else 0.5, device="cuda")
    h, vmax = (10.0, 2500.0) if physics == "velocity" else (2e-3, 509.8366)
    m = W.Model(p, h, O.cfl_dt(h, vmax, 2, order, 0.5), order, physics)
    rec = torch.arange(max(4, int(dense * n)), device="cuda")
    arr, o = W._shot_descs([W.Shot(n - 1, torch.ones(nt + 1, device="cuda"), rec)]), W.GradOpts()
    o.mode, o.k = W.MODE[mode], 1.0
    full, least = W._sz(0), W._sz(0)
    assert W._grad_ws(m._h, arr, 1, W.C.byref(o), W.C.byref(full)) == 0
    assert W._grad_min(m._h, arr, 1, W.C.byref(o), W.C.byref(least)) == 0
    assert (full.value > least.value) == several
