"""Kernel variants at the sizes where one takes over from another: depth kernels, column and row
passes, folded direct DFTs, surface transforms and the contact solvers, each against the FP64
oracle at the bars of the operators (relative L2 1e-10 in FP64, 2e-5 in FP32) and of the contact
solve (pressure 1e-9 in FP64 with both sides converged to 1e-13, 2e-5 in FP32)."""
import numpy as np
import pytest

from oracle import contact as C
from oracle import operators as op
from oracle import tensors as T
from paper_1811_11558_gb300 import inputs

from gpu_util import rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu

E, NU = 1.0, 0.3
ES = T.e_star(E, NU)
TOL = {"fp64": 1e-10, "fp32": 2e-5}


def _ctx(n1, n2, z, prec, L2=1.0, **kw):
    from paper_1811_11558_gb300 import Context

    return Context(n1, n2, z, 1.0, L2, precision=prec, E=E, nu=NU, **kw)


def _refined(nz, depth):
    return depth * np.linspace(0.0, 1.0, nz) ** 1.5


@pytest.mark.parametrize("n1,n2,z,prec", [
    (32, 16, inputs.uniform_depth(2, 0.1), "fp32"),      # two nodes, one chunk: no carries
    (32, 16, _refined(3, 0.1), "fp64"),
    (32, 16, _refined(33, 0.3), "fp32"),                  # last chunk of one node
    (16, 16, _refined(47, 0.4), "fp64"),                  # chunks of three, ragged
    (16, 8, inputs.uniform_depth(140, 0.4), "fp64"),      # nine nodes per chunk: local terms in shared memory
    (128, 256, inputs.uniform_depth(5, 0.02), "fp64"),    # rows with the three pair transforms in one thread
    (64, 1024, inputs.uniform_depth(2, 0.004), "fp32"),   # columns of 1024 points, 8 per CTA
    (3, 3, inputs.uniform_depth(4, 0.2), "fp64"),         # smallest direct DFT, odd and even sides
    (4, 3, _refined(5, 0.2), "fp32"),
    (255, 5, inputs.uniform_depth(2, 0.01), "fp64"),      # longest direct DFT
    (7, 256, inputs.uniform_depth(2, 0.01), "fp32"),
])
@pytest.mark.parametrize("kind", ["stress", "strain"])
def test_mindlin_variants(n1, n2, z, prec, kind):
    torch = require_gpu()
    ep = inputs.plastic_strain_field(n1, n2, z, seed=41 + n1 + n2 + z.size)
    ref, u3_ref = op.mindlin_apply(ep, z, 1.0, 0.9, E, NU, kind, with_surface=True)
    ctx = _ctx(n1, n2, z, prec, L2=0.9)
    u3 = torch.empty(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
    out = ctx.apply_mindlin(to_dev(torch, ep, ctx.dtype), kind=kind, u3=u3)
    torch.cuda.synchronize()
    assert rel_l2(out.cpu().numpy(), ref) < TOL[prec]
    assert rel_l2(u3.cpu().numpy(), u3_ref) < TOL[prec]


def test_cutoff_on_a_refined_grid():
    """Neighbour carries under the cutoff (no carry recurrence) against the exact scan on refined
    nodes: the dropped terms are below e^-18 of the moments, at the FP32 rounding level."""
    torch = require_gpu()
    z = _refined(32, 2.0)                                  # every chunk span beyond the cutoff for |k| > ~100
    ep = inputs.plastic_strain_field(512, 64, z, seed=43, z_decay=1.0)
    ctx = _ctx(512, 64, z, "fp32", L2=0.125)
    d = to_dev(torch, ep, torch.float32)
    u3 = torch.empty(ctx.surf_shape, dtype=torch.float32, device="cuda")
    outs = {}
    for eps in (0.0, 18.0):
        ctx.set_plan(4, depth_cutoff=eps)
        outs[eps] = [ctx.apply_mindlin(d, u3=u3).cpu().numpy().astype(np.float64), u3.cpu().numpy().astype(np.float64)]
    for a, b in zip(outs[18.0], outs[0.0]):
        assert rel_l2(a, b) < 1e-6


@pytest.mark.parametrize("nu", [-0.5, 0.0, 0.49])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_mindlin_material_range(prec, nu):
    """The moments' constants over the range of Poisson's ratio (2 nu - 1 and 1 - nu vary)."""
    torch = require_gpu()
    from paper_1811_11558_gb300 import Context

    z = inputs.uniform_depth(9, 0.3)
    ep = inputs.plastic_strain_field(32, 16, z, seed=44)
    ctx = Context(32, 16, z, 1.0, 1.0, precision=prec, E=2.0, nu=nu)
    for kind in ("stress", "strain"):
        ref = op.mindlin_apply(ep, z, 1.0, 1.0, 2.0, nu, kind)
        out = ctx.apply_mindlin(to_dev(torch, ep, ctx.dtype), kind=kind)
        torch.cuda.synchronize()
        assert rel_l2(out.cpu().numpy(), ref) < TOL[prec]


@pytest.mark.parametrize("n1,n2,prec", [(16, 1024, "fp32"), (1024, 16, "fp64"), (16, 2, "fp32"), (8, 64, "fp64"),
                                        (64, 64, "fp32"), (1024, 64, "fp32")])
def test_surface_transforms(n1, n2, prec):
    """Pressure to surface displacement and volume field at the smallest and largest sides of the
    surface transforms and of the column pass that evaluates the field."""
    torch = require_gpu()
    z = inputs.uniform_depth(2, 0.01)
    p = np.abs(inputs.random_field((n2, n1), seed=45 + n1)) + 0.5
    for kind in ("stress", "strain"):
        u3_ref, vol_ref = op.boussinesq_apply(p, z, 1.0, 0.8, E, NU, kind)
        ctx = _ctx(n1, n2, z, prec, L2=0.8)
        d = to_dev(torch, p, ctx.dtype)
        u3 = torch.empty(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
        vol = torch.empty(ctx.vol_shape, dtype=ctx.dtype, device="cuda")
        ctx.apply_boussinesq(d, u3=u3, vol=vol, kind=kind)
        only = torch.empty_like(vol)
        ctx.apply_boussinesq(d, vol=only, kind=kind)
        torch.cuda.synchronize()
        assert rel_l2(u3.cpu().numpy(), u3_ref) < TOL[prec]
        assert rel_l2(vol.cpu().numpy(), vol_ref) < TOL[prec]
        assert torch.equal(only, vol)


@pytest.mark.parametrize("n1,n2,prec", [(16, 16, "fp64"), (16, 16, "fp32"), (32, 32, "fp32"), (64, 64, "fp64"),
                                        (128, 128, "fp64"), (128, 128, "fp32"),          # one cluster
                                        (32, 16, "fp64"), (16, 64, "fp32"), (256, 32, "fp64"),  # six kernels
                                        (8, 16, "fp64"), (27, 21, "fp64")])              # sides without a variant
def test_contact_variants(n1, n2, prec):
    """Elastic contact on every path against the oracle, from a zero and from a given guess; an
    iteration cap is reported; a non-finite surface is refused and the context stays usable."""
    torch = require_gpu()
    from paper_1811_11558_gb300 import FvimError

    z = inputs.uniform_depth(2, 0.1)
    h = inputs.hertz_profile(n1, n2, 1.0, 1.0, 0.5)
    W = 2e-2 * ES * (np.pi / 4) ** 2
    ref, _ = C.polonsky_keer(h, W, 1.0, 1.0, E, NU, tol=1e-13)
    ctx = _ctx(n1, n2, z, prec)
    dt = ctx.dtype
    hd = to_dev(torch, h, dt)
    opts = ctx.default_opts(cg_tol=1e-13) if prec == "fp64" else ctx.default_opts()
    tol = 1e-9 if prec == "fp64" else 2e-5
    p = torch.zeros(ctx.surf_shape, dtype=dt, device="cuda")
    it, err = ctx.elastic_contact(hd, W, p, opts)
    assert err < opts.cg_tol and rel_l2(p.cpu().numpy(), ref) < tol
    guess = p * 0.5 + 1e-3
    ctx.elastic_contact(hd, W, guess, opts)
    assert rel_l2(guess.cpu().numpy(), ref) < tol
    assert abs(float(guess.double().mean()) - W) < (1e-13 if prec == "fp64" else 1e-6) * W * 10
    it, err = ctx.elastic_contact(hd, W, torch.zeros_like(p), ctx.default_opts(cg_max_iter=3), allow_not_converged=True)
    assert it == 3
    bad = hd.clone()
    bad[n2 - 1, n1 - 1] = float("nan")
    with pytest.raises(FvimError):
        ctx.elastic_contact(bad, W, torch.zeros_like(p), opts)
    again = torch.zeros_like(p)
    ctx.elastic_contact(hd, W, again, opts)
    assert torch.equal(again, p)


@pytest.mark.parametrize("hole", [1e6, 1e12, 1e20, 1e30])
@pytest.mark.parametrize("n1,n2", [(16, 16), (64, 64), (64, 32), (256, 256)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_contact_with_a_masked_point(n1, n2, prec, hole):
    """A point far below the surface dominates the first mean gap and never carries load: the
    pressure is that of a hole just deep enough not to touch, whatever its depth."""
    torch = require_gpu()
    z = inputs.uniform_depth(2, 0.1)
    h = inputs.hertz_profile(n1, n2, 1.0, 1.0, 0.5)
    W = 2e-2 * ES * (np.pi / 4) ** 2
    h[1, 2] = -10.0
    ref, _ = C.polonsky_keer(h, W, 1.0, 1.0, E, NU, tol=1e-13)
    assert ref[1, 2] == 0
    h[1, 2] = -hole
    ctx = _ctx(n1, n2, z, prec)
    opts = ctx.default_opts(cg_tol=1e-13) if prec == "fp64" else ctx.default_opts()
    p = torch.zeros(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
    ctx.elastic_contact(to_dev(torch, h, ctx.dtype), W, p, opts)
    assert rel_l2(p.cpu().numpy(), ref) < (1e-9 if prec == "fp64" else 2e-5)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_contact_loop_equals_batches(prec, monkeypatch):
    """The six-kernel iteration as one WHILE graph and as host-driven batches: the same bits, for two
    surfaces, loads and pressures through one context (they live in the device state)."""
    torch = require_gpu()
    z = inputs.uniform_depth(2, 0.1)
    res = {}
    for mode in ("1", "0"):
        monkeypatch.setenv("FVIM_DEVICE_CG", mode)
        ctx = _ctx(64, 32, z, prec, L2=0.5)
        res[mode] = []
        for R, W in ((0.5, 2e-3), (0.3, 5e-3)):
            h = to_dev(torch, inputs.hertz_profile(64, 32, 1.0, 0.5, R), ctx.dtype)
            p = torch.zeros(ctx.surf_shape, dtype=ctx.dtype, device="cuda")
            res[mode].append((ctx.elastic_contact(h, W, p), p.cpu().numpy()))
        ctx.close()
    for a, b in zip(res["1"], res["0"]):
        assert a[0] == b[0] and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("n1,n2,nz", [(16, 4, 6), (64, 32, 5)])
def test_plastic_increment_fp32_sums(n1, n2, nz):
    """FP32 residual sums by whole planes, at planes shorter and longer than a block."""
    torch = require_gpu()
    z = inputs.uniform_depth(nz, 0.4)
    x = (np.arange(n1) + 0.5) / n1 - 0.5
    y = (np.arange(n2) + 0.5) / n2 - 0.5
    dT = 0.15 * ES * np.sqrt(np.maximum(0.0, 1.0 - (x[None, :] ** 2 + y[:, None] ** 2) / 0.09))
    sy, Eh = 0.05 * ES, 0.1
    ref = C.plasticity_solve(dT, C.PlasticState(nz, n2, n1), z, 1.0, 1.0, E, NU, sy, Eh, tol_rel=1e-13)
    assert ref[2].max() > 0
    ctx = _ctx(n1, n2, z, "fp32", sigma_y=sy, E_h=Eh)
    out = [torch.empty(s, dtype=torch.float32, device="cuda") for s in (ctx.vol_shape, ctx.vol_shape, ctx.scal_shape)]
    ctx.plasticity_solve(to_dev(torch, dT, torch.float32), *out)
    for got, want, f in zip(out, ref, (1, 10, 10)):
        assert rel_l2(got.cpu().numpy(), want) < 2e-5 * f
