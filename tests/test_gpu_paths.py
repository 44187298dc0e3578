"""GPU paths that a call takes by its size: the default lane count against the
lane count whose summation order it keeps, taped rollouts whose step records
run out, the right-hand sides with contacts from distance of recorded steps,
and the parameter gradients of environments without contact."""

import numpy as np
import pytest

from paper_2506_14186_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dmx():
    import torch
    from paper_2506_14186_gb300 import _build
    _build.build()
    import paper_2506_14186_gb300 as d
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return d


def _dev(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _call(dmx, model, inp, **kw):
    ctrl = None if inp["ctrl"] is None else _dev(np.transpose(inp["ctrl"], (1, 2, 0)))
    args = dict(NI=inp["NI"], rtol=inp["rtol"], atol=inp["atol"], h0=inp["h0"], max_steps=4000)
    args.update(kw)
    return dmx.rollout(model, _dev(inp["x0"].T), _dev(inp["T"]), ctrl=ctrl, **args)


# the fewest lanes that give each of the GPU's 608 sub-partitions a warp at these batch sizes
@pytest.mark.parametrize("name,B,lanes", [("ball", 19457, 1), ("box", 9729, 2), ("box", 4865, 4), ("box", 1, 32),
                                          ("quadruped", 2433, 8), ("chain_cube", 1217, 16)])
def test_default_lanes_keep_the_step_decisions(dmx, name, B, lanes):
    """Without a lane count the call runs on as many lanes as fill the SMs but
    sums the error norm in the order of `lanes`: the same bits."""
    import torch
    inp = W.INPUTS[name](B) if name == "quadruped" else W.INPUTS[name](B, T=0.01)
    if name == "quadruped":
        inp["x0"][:, 2] = 0.427
    inp["T"] = np.full(B, 0.01)
    model = dmx.Model(W.SCENES[name]())
    a = _call(dmx, model, inp)
    b = _call(dmx, model, inp, lanes=lanes)
    for k in ("xT", "nsteps", "nrej", "status"):
        assert torch.equal(a[k], b[k]), k


def test_records_that_run_out(dmx):
    """A tape holds records for 512 steps an environment on average; later
    segments are recomputed.  Both give the gradient that recomputing every
    segment gives (the same right-hand sides, so within rounding of it)."""
    import torch
    sc, inp = W.box_scene(), W.box_push_inputs(3, seed=5, T=0.12)
    inp["rtol"], inp["atol"] = 1e-9, 1e-11
    bar = _dev(np.random.default_rng(2).normal(size=(13, 3)))
    got = {}
    for mode in ("reverse", "recompute"):
        model = dmx.Model(sc)
        model.set_adjoint(mode)
        out = _call(dmx, model, inp, tape=True, K=32)
        got[mode] = dmx.rollout_grad(out["tape"], bar)[0]
        steps = int(out["nsteps"].sum())
    assert steps > 3 * 512, steps
    scale = got["recompute"].abs().amax(0)
    assert float(((got["reverse"] - got["recompute"]).abs() / scale).max()) < 1e-12
    assert torch.isfinite(got["reverse"]).all()


@pytest.mark.parametrize("name,B,T,NI,method", [("box", 5, 0.02, 1, "dopri5"), ("box", 70, 0.02, 1, "euler"),
                                                 ("quadruped", 3, 0.02, 1, "tsit5"), ("chain_cube", 2, 0.04, 3, "dopri5")])
def test_cfd_stages_of_recorded_steps(dmx, name, B, T, NI, method):
    """With contacts from distance the right-hand sides at the recorded stage
    states are evaluated beforehand; the gradient is that of evaluating them
    in the sweep (within 1e-9: the same formulas along the same steps)."""
    sc = W.SCENES[name](**W.CFD_OPTIONS)
    inp = W.chain_inputs(B, T=T, NI=NI) if name == "chain_cube" else W.INPUTS[name](B)
    inp["T"] = np.full(B, T)
    if name == "quadruped":
        inp["x0"][:, 2] = 0.4255
    model = dmx.Model(sc)
    bar = _dev(np.random.default_rng(6).normal(size=(model.nx, B)))
    out = _call(dmx, model, inp, tape=True, K=8, method=method)
    got = {}
    for mode in ("reverse", "recompute"):
        model.set_adjoint(mode)
        got[mode] = dmx.rollout_grad(out["tape"], bar, cfd=True)
    for a, b in zip(got["reverse"], got["recompute"]):
        if b is not None and b.numel():
            assert float((a - b).abs().max()) <= 1e-9 * float(b.abs().max())


@pytest.mark.parametrize("name,B", [("ball", 1), ("ball", 65), ("toss", 33)])
def test_parameter_gradients_without_contact(dmx, name, B):
    """Environments that met no contact keep the forward-mode kernel's
    parameter gradients bit for bit, whatever else the batch holds."""
    import torch
    sc = W.box_scene(solref=(0.005, 1.0)) if name == "toss" else W.SCENES[name]()
    inp = W.INPUTS[name](B, T=0.05)
    ground = np.arange(B) % 2 == 1        # every other one falls onto the plane from below its rest height
    inp["x0"][:, 2] = np.where(ground, 0.045 if name == "toss" else 0.095, 2.0 + 0.01 * np.arange(B))
    inp["x0"][:, 9] = np.where(ground, -0.5, 0.0)
    model = dmx.Model(sc)
    bar = _dev(np.random.default_rng(4).normal(size=(model.nx, B)))
    out = _call(dmx, model, inp, tape=True, K=8)
    res = {}
    for mode in ("reverse", "recompute", "tangent"):
        model.set_adjoint(mode)
        res[mode] = dmx.rollout_grad_params(out["tape"], bar)
    for k in (0, 2):
        for mode in ("reverse", "recompute"):
            a, b = res[mode][k], res["tangent"][k]
            assert torch.equal(a[:, ::2], b[:, ::2]), (k, mode)
            assert torch.isfinite(a).all()
    if B > 1:                              # the ones on the ground have a gradient, by the reverse-mode kernel
        assert float(res["reverse"][2][:, 1::2].abs().amax(0).min()) > 1e-6
