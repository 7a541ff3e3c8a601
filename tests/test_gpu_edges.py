"""Limits of the solvers and operators that the oracle comparisons do not reach: iteration caps,
non-finite input, deep grids, launch plans and selection switches."""
import numpy as np
import pytest

from oracle import tensors as T
from paper_1811_11558_gb300 import inputs

from gpu_util import rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu

E, NU = 1.0, 0.3
ES = T.e_star(E, NU)


def _ctx(n1, n2, z, prec, **kw):
    from paper_1811_11558_gb300 import Context

    kw = {"E": E, "nu": NU, **kw}
    return Context(n1, n2, z, 1.0, 1.0, precision=prec, **kw)


def _hertz(torch, ctx, R=0.5):
    h = to_dev(torch, inputs.hertz_profile(ctx.n1, ctx.n2, 1.0, 1.0, R), ctx.dtype)
    return h, 2e-2 * ES * (np.pi / 4) ** 2


@pytest.mark.parametrize("loop", ["1", "0"])
def test_contact_loop_ends_at_the_iteration_cap(loop, monkeypatch):
    """The loop of a power-of-two surface stops after cg_max_iter passes with that count, also after a
    refused solve, and on a side stream from a context's first solve on (the arrival counter of its sums is
    cleared by every solve on the solver's own stream)."""
    torch = require_gpu()
    monkeypatch.setenv("FVIM_DEVICE_CG", loop)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = _ctx(256, 64, inputs.uniform_depth(2, 0.1), "fp32")
        h, W = _hertz(torch, ctx)
        bad = h.clone()
        bad[3, 5] = float("nan")
        for cap in (1, 2, 5, 3):
            it, err = ctx.elastic_contact(h, W, torch.zeros_like(h), ctx.default_opts(cg_tol=1e-30, cg_max_iter=cap),
                                          allow_not_converged=True)
            assert it == cap and np.isfinite(err)
            with pytest.raises(Exception):
                ctx.elastic_contact(bad, W, torch.zeros_like(h), ctx.default_opts(cg_max_iter=cap))
    side.synchronize()


def test_dfsane_loop_ends_at_its_caps():
    """The device loop of a plastic increment stops after df_max_iter accepted points, reported as not
    converged, and a later solve through the same context is that of a fresh one."""
    torch = require_gpu()
    from paper_1811_11558_gb300 import FvimError

    z = inputs.uniform_depth(6, 0.4)
    sy = 0.05 * ES
    x = (np.arange(32) + 0.5) / 32 - 0.5
    p = 0.15 * ES * np.sqrt(np.maximum(0.0, 1.0 - (x[None, :] ** 2 + x[:, None] ** 2) / 0.09))

    def solve(ctx, **kw):
        out = [torch.empty(s, dtype=ctx.dtype, device="cuda") for s in (ctx.vol_shape, ctx.vol_shape, ctx.scal_shape)]
        rep = ctx.plasticity_solve(to_dev(torch, p, ctx.dtype), *out, ctx.default_opts(**kw))
        torch.cuda.synchronize()
        return rep, out

    for prec in ("fp32", "fp64"):
        ctx = _ctx(32, 32, z, prec, sigma_y=sy, E_h=0.1)
        full, ref = solve(ctx)
        for cap in (1, 2):
            assert cap < full[0]
            with pytest.raises(FvimError, match="not converged"):
                solve(ctx, df_max_iter=cap)
        again, out = solve(ctx)
        assert again == full and all(torch.equal(a, b) for a, b in zip(out, ref))


@pytest.mark.parametrize("n1,nz", [(32, 512), (32, 256), (8, 128)])
def test_deep_uniform_grids_propagate_without_drift(n1, nz):
    """FP32 against FP64 far below a smooth plastic strain at the surface, on uniform grids that take the
    shared-memory depth kernel.  Bar: a propagator over a chunk of C nodes is a power, C - 1 roundings
    of the element's; the carry to the last of nch chunks takes nch more, source, moments, output and
    transforms fewer than ten: (C + nch + 10) 2^-24 in all (3.5e-6 at 512 nodes).  A power over the whole
    depth would take nz roundings of one sign."""
    torch = require_gpu()
    depth = 0.1
    z = inputs.uniform_depth(nz, depth)
    x, y = np.arange(n1) / n1, np.arange(32) / 32
    ep = np.zeros((nz, 6, 32, n1))
    rng = np.random.default_rng(n1 + nz)
    for k1, k2 in ((1, 0), (0, 1), (1, 1), (1, 2), (2, 1), (2, 2), (2, 3), (1, 3), (0, 3), (0, 2)):
        ph = 2 * np.pi * (k1 * x[None, :] + k2 * y[:, None])
        a = rng.standard_normal((2, 6, 1, 1)) * 1e-3
        ep[:2] += a[0] * np.cos(ph) + a[1] * np.sin(ph)
    out = {}
    for prec in ("fp64", "fp32"):
        ctx = _ctx(n1, 32, z, prec)
        out[prec] = ctx.apply_mindlin(to_dev(torch, ep, ctx.dtype)).cpu().numpy().astype(np.float64)
    C = ctx.plan["depth_chunk"]
    bar = (C + -(-nz // C) + 10) * 2.0 ** -24
    last = slice(nz - C, nz)
    assert rel_l2(out["fp32"][last], out["fp64"][last]) < bar


@pytest.mark.parametrize("n1,n2,nz", [(16, 8, 37), (4, 4, 23), (64, 4, 150)])
@pytest.mark.parametrize("refined", [False, True])
def test_chunk_lengths_agree_in_the_shared_memory_kernel(n1, n2, nz, refined):
    """Every accepted chunk length, odd and even, with a ragged last chunk and tiles of every width: the
    same operator to the rounding of FP64 (1e-13 of it), and FP32 within the operator's bar of FP64."""
    torch = require_gpu()
    from paper_1811_11558_gb300 import FvimError

    z = 0.3 * np.linspace(0.0, 1.0, nz) ** (1.5 if refined else 1.0)
    ep = inputs.plastic_strain_field(n1, n2, z, seed=48)
    ref = None
    for prec, chunks in (("fp64", range(2, 20)), ("fp32", range(9, 20))):
        ctx = _ctx(n1, n2, z, prec)
        d = to_dev(torch, ep, ctx.dtype)
        ran = []
        for C in chunks:
            try:
                ctx.set_plan(C)
            except FvimError:
                continue
            u3 = torch.empty(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
            out = [t.cpu().numpy().astype(np.float64) for t in (ctx.apply_mindlin(d, u3=u3), u3)]
            if ref is None:
                ref = out
            assert all(rel_l2(a, b) < (1e-13 if prec == "fp64" else 2e-5) for a, b in zip(out, ref)), (prec, C)
            ran.append(C)
        assert len(ran) > 6


@pytest.mark.parametrize("n1,n2", [(64, 64), (64, 32)])       # one cluster; six kernels
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_contact_refuses_infinite_input(n1, n2, prec):
    """An infinite height above a point without starting pressure re-enters the contact with an infinite
    pressure, an infinite starting pressure leaves no contact: both are refused.  An infinite depth below
    such a point is a hole like any other."""
    torch = require_gpu()
    from paper_1811_11558_gb300 import FvimError

    ctx = _ctx(n1, n2, inputs.uniform_depth(2, 0.1), prec)
    h, W = _hertz(torch, ctx)
    guess = torch.ones_like(h)
    guess[1, 2] = 0
    up = h.clone()
    up[1, 2] = float("inf")
    with pytest.raises(FvimError, match="non-finite"):
        ctx.elastic_contact(up, W, guess.clone())
    inf = guess.clone()
    inf[n2 // 2, n1 // 2] = float("inf")
    with pytest.raises(FvimError, match="non-finite"):
        ctx.elastic_contact(h, W, inf)
    res = []
    for depth in (float("-inf"), -10.0):
        down, p = h.clone(), guess.clone()
        down[1, 2] = depth
        ctx.elastic_contact(down, W, p)
        assert p[1, 2] == 0
        res.append(p.cpu().numpy().astype(np.float64))
    assert rel_l2(res[0], res[1]) < (1e-9 if prec == "fp64" else 2e-5)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_small_contact_without_the_cluster(prec, monkeypatch):
    """The six kernels take over on the surfaces of the cluster kernel (FVIM_CONTACT_CLUSTER=0, or a refused
    launch): the same pressure at the bar of the contact solve, not the same bits (the sums add up in
    another order)."""
    torch = require_gpu()
    ctx = _ctx(64, 64, inputs.uniform_depth(2, 0.1), prec)
    h = to_dev(torch, inputs.self_affine_surface(64, 1.0, 0.8, 4, 8, 16, 0.1, seed=7), ctx.dtype)
    W = 2e-2 * ES * 0.1
    opts = ctx.default_opts(cg_tol=1e-13) if prec == "fp64" else ctx.default_opts()
    p = {}
    for mode in ("1", "0"):
        monkeypatch.setenv("FVIM_CONTACT_CLUSTER", mode)
        p[mode] = torch.zeros_like(h)
        ctx.elastic_contact(h, W, p[mode], opts)
    assert not torch.equal(p["0"], p["1"])
    a, b = (p[m].cpu().numpy().astype(np.float64) for m in "01")
    assert rel_l2(a, b) < (1e-9 if prec == "fp64" else 2e-5)


def test_three_cta_plans_run_where_their_tile_fits_thrice():
    """A plan for three CTAs per SM is accepted on refined nodes as on uniform ones; where the element
    table of the refined grid takes the room, it runs and reports two, and the tuner does not time it."""
    torch = require_gpu()
    uni = inputs.uniform_depth(64, 0.4)
    ref = 0.4 * np.linspace(0.0, 1.0, 64) ** 1.5
    short = 0.4 * np.linspace(0.0, 1.0, 32) ** 1.5
    for z, ctas in ((uni, 3), (ref, 2), (short, 3)):
        ctx = _ctx(128, 32, z, "fp32")
        d = to_dev(torch, inputs.plastic_strain_field(128, 32, z, seed=47), torch.float32)
        ctx.set_plan(4, depth_ctas=2)
        two = ctx.apply_mindlin(d).cpu().numpy()
        ctx.set_plan(4, depth_ctas=3)
        assert ctx.plan["depth_ctas"] == ctas
        three = ctx.apply_mindlin(d).cpu().numpy()
        assert rel_l2(three, two) < 1e-6
        assert (4 in ctx.autotune(reps=3).get("timings_ms_3ctas", {})) == (ctas == 3)


@pytest.mark.parametrize("n1,n2,nz", [(3, 3, 2), (255, 2, 2), (256, 3, 2), (3, 256, 2), (4, 255, 2), (33, 7, 3)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_direct_transforms_at_their_limits(n1, n2, nz, prec):
    """Direct DFTs of the shortest and longest sides next to short ones (few rows, columns and CTAs), through
    the operator and the surface convolution, at the operators' bars."""
    torch = require_gpu()
    from oracle import operators as op

    z = inputs.uniform_depth(nz, 0.02)
    ep = inputs.plastic_strain_field(n1, n2, z, seed=49)
    p = np.abs(inputs.random_field((n2, n1), seed=50)) + 0.5
    ref, u3_ref = op.mindlin_apply(ep, z, 1.0, 1.0, E, NU, "stress", with_surface=True)
    ctx = _ctx(n1, n2, z, prec)
    u3 = torch.empty(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
    out = ctx.apply_mindlin(to_dev(torch, ep, ctx.dtype), u3=u3)
    bu = torch.empty_like(u3)
    ctx.apply_boussinesq(to_dev(torch, p, ctx.dtype), u3=bu)
    tol = 1e-10 if prec == "fp64" else 2e-5
    assert rel_l2(out.cpu().numpy(), ref) < tol and rel_l2(u3.cpu().numpy(), u3_ref) < tol
    assert rel_l2(bu.cpu().numpy(), op.boussinesq_apply(p, z, 1.0, 1.0, E, NU, "stress")[0]) < tol


def test_first_solve_on_a_side_stream():
    """A context's first solve fills its workspace; on a stream that does not wait for the legacy one it gives
    the bits of a later solve."""
    torch = require_gpu()
    z = inputs.uniform_depth(24, 0.3)
    sy = 0.05 * ES
    x = (np.arange(256) + 0.5) / 256 - 0.5
    p = 0.13 * ES * np.sqrt(np.maximum(0.0, 1.0 - (x[None, :] ** 2 + x[:, None] ** 2) / 0.06))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = _ctx(256, 256, z, "fp32", sigma_y=sy, E_h=0.1)
        d = to_dev(torch, p, torch.float32)
        res = []
        for _ in range(2):
            out = [torch.empty(s, dtype=ctx.dtype, device="cuda") for s in (ctx.vol_shape, ctx.vol_shape, ctx.scal_shape)]
            res.append((ctx.plasticity_solve(d, *out), out))
    side.synchronize()
    assert res[0][0] == res[1][0] and all(torch.equal(a, b) for a, b in zip(res[0][1], res[1][1]))
