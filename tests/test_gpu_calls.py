"""Calls whose lanes, memory or device work follow a rule: the lane count that
a model names, step records, and what is given back."""

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


def _inputs(name, B, T, NI=1, seed=0):
    inp = (W.chain_inputs(B, seed=seed, T=T, NI=NI) if name == "chain_cube" else
           W.INPUTS[name](B, seed=seed))
    inp["T"] = np.full(B, T)
    if name == "quadruped":
        inp["x0"][:, 2] = 0.427
    return inp


def _call(dmx, model, inp, **kw):
    ctrl = None if inp["ctrl"] is None else _dev(np.transpose(inp["ctrl"], (1, 2, 0)))
    args = dict(NI=inp["NI"], rtol=inp["rtol"], atol=inp["atol"], h0=inp["h0"], max_steps=4000)
    args.update(kw)
    return dmx.rollout(model, _dev(inp["x0"].T), _dev(inp["T"]), ctrl=ctrl, **args)


# batches where the lanes of the summation order and those of the call are different
@pytest.mark.parametrize("name,B,T", [("ball", 20000, 0.1), ("box", 5000, 0.03), ("quadruped", 2500, 0.01),
                                      ("box", 3, 0.02)])
@pytest.mark.parametrize("recorded", [0, 8])
def test_the_lanes_a_model_names_give_the_same_bits(dmx, name, B, T, recorded):
    """Model.lanes(B), passed as lanes, gives the bits of the call without lanes,
    whether a lane count is recorded or not."""
    import torch
    model = dmx.Model(W.SCENES[name]())
    if recorded:
        model.set_lanes(B, recorded)
    inp = _inputs(name, B, T)
    a = _call(dmx, model, inp)
    b = _call(dmx, model, inp, lanes=model.lanes(B))
    for k in ("xT", "nsteps", "nrej", "status"):
        assert torch.equal(a[k], b[k]), k
