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


# fixed steps: batches a little over the warps that an SM's registers hold
@pytest.mark.parametrize("name,B", [("billiard", 2000), ("billiard", 4096), ("capsules", 1900), ("chain_cube", 1400)])
def test_lanes_of_fixed_step_rollouts_keep_the_results(dmx, name, B):
    import torch
    model = dmx.Model(W.SCENES[name]())
    inp = _inputs(name, B, 0.02)
    a = _call(dmx, model, inp, method="euler")
    b = _call(dmx, model, inp, method="euler", lanes=32)
    for k in ("xT", "nsteps", "status"):
        assert torch.equal(a[k], b[k]), k


# ------------------------------------------------------------------ step records: memory
_MEMORY = r'''
import ctypes, gc, re, sys
import numpy as np, torch
from paper_2506_14186_gb300 import workloads as W
import paper_2506_14186_gb300 as dmx

rt = ctypes.CDLL(next(l.split()[-1] for l in open("/proc/self/maps") if re.search(r"libcudart\.so", l)))
torch.zeros(1, device="cuda")
pool = ctypes.c_void_p()
assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0

def used():                                     # bytes of the device's default pool in use (attribute 7)
    torch.cuda.synchronize()
    v = ctypes.c_uint64()
    assert rt.cudaMemPoolGetAttribute(pool, 7, ctypes.byref(v)) == 0
    return v.value

def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]

def dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")

def tape(model, inp, T, **kw):
    B = len(inp["x0"])
    ctrl = None if inp["ctrl"] is None else dev(np.transpose(inp["ctrl"], (1, 2, 0)))
    return dmx.rollout(model, dev(inp["x0"].T), dev(np.full(B, T)), ctrl=ctrl, NI=inp["NI"], max_steps=2000,
                       tape=True, **kw)["tape"]

GiB = 1 << 30
'''


def _run(code):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _MEMORY + code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


def test_records_do_not_depend_on_what_the_pool_keeps_unused(dmx):
    """With little memory free, a tape gets the same room as the one freed before
    it: the pool's unused bytes count as free."""
    _run(r'''
model, inp = dmx.Model(W.box_scene()), W.box_push_inputs(20000)
filler = torch.empty(free() - 80 * GiB, dtype=torch.uint8, device="cuda")
sizes = []
for _ in range(3):
    t = tape(model, inp, 0.001, K=8)
    assert used() > 6 * GiB, used() / GiB
    sizes.append(used())
    del t; gc.collect()
    assert used() < GiB
assert max(sizes) - min(sizes) < GiB // 8, sizes
''')


def test_live_tapes_hold_a_bounded_amount_of_records(dmx):
    """Tapes that want 24 GiB of step records each hold 48 GiB together at most
    (a tape's own arrays: below 1 GiB here)."""
    _run(r'''
model, inp = dmx.Model(W.box_scene()), W.box_push_inputs(20000)
tapes = [tape(model, inp, 0.001) for _ in range(4)]
full = used()
assert 24 * GiB < full < (48 + 4) * GiB, full / GiB
del tapes[0]; gc.collect()
assert used() < full - 12 * GiB
tapes.append(tape(model, inp, 0.001))           # the room of a freed tape can be had again
assert abs(used() - full) < GiB, (used() / GiB, full / GiB)
''')


def test_no_records_that_complete_no_segment(dmx):
    """Records that could not hold one segment of every environment are
    not kept (2048 arms, 2.5 GiB: 11 steps of 118 KB an arm)."""
    _run(r'''
model, inp = dmx.Model(W.SCENES["chain_cube"]()), W.chain_inputs(2048, T=0.001)
filler = torch.empty(free() - 20 * GiB, dtype=torch.uint8, device="cuda")
t = tape(model, inp, 0.001, K=64)
assert used() < GiB // 2, used() / GiB
del t; gc.collect()
t = tape(model, inp, 0.001, K=8)                # the first segment: kept
assert used() > GiB, used() / GiB
''')


def test_the_last_model_gives_back_the_memory(dmx):
    """What the pool keeps of freed tapes goes back to the device with the last model."""
    _run(r'''
before = free()
model, inp = dmx.Model(W.box_scene()), W.box_push_inputs(20000)
other = dmx.Model(W.SCENES["ball"]())
t = tape(model, inp, 0.001)
assert before - free() > 16 * GiB
del t, model; gc.collect()
del other; gc.collect()
assert before - free() < GiB, (before - free()) / GiB
''')


# ------------------------------------------------------------------ step records: results
@pytest.mark.parametrize("cfd", [False, True])
def test_repeated_calls_with_too_few_records(dmx, cfd):
    """Capsules resting with contact rows at the edge of the active set: where the
    Newton search starts decides their last bits, so a kept and a recomputed
    segment differ there.  Which segments are kept when there is little memory
    must not depend on scheduling: the same call gives the same bits again."""
    _run(r'''
cfd = %r
model, inp = dmx.Model(W.SCENES["capsules"](**(W.CFD_OPTIONS if cfd else {}))), W.INPUTS["capsules"](2000)
bar = dev(np.random.default_rng(8).normal(size=(model.nx, 2000)))
filler = torch.empty(free() - 24 * GiB, dtype=torch.uint8, device="cuda")
first = None
for k in range(5):
    t = tape(model, inp, 0.1, K=8, rtol=inp["rtol"], atol=inp["atol"], h0=inp["h0"])
    n = t.read()[1]
    g = dmx.rollout_grad(t, bar, cfd=cfd)[0]
    assert used() > 2 * GiB and int(n.max()) > 64   # records, and more steps than they hold
    del t; gc.collect()
    assert torch.isfinite(g).all()
    first = g if first is None else first
    assert torch.equal(first, g), (k, int((first != g).any(0).sum()))
''' % cfd)


@pytest.mark.parametrize("B", [1, 3, 1500])
def test_cfd_stages_over_uneven_step_counts(dmx, B):
    """The recorded steps that are evaluated beforehand are numbered without gaps
    over environments with many, few and no steps (a state that is not finite
    takes none: its cotangent passes through)."""
    import torch
    model = dmx.Model(W.box_scene(**W.CFD_OPTIONS))
    inp = W.box_push_inputs(B, seed=3, T=0.01)
    inp["T"] = 0.012 * (1 + np.arange(B) % 7) / 7.0
    if B > 1:
        inp["x0"][1::5, 0] = np.nan
    bar = _dev(np.random.default_rng(6).normal(size=(model.nx, B)))
    out = _call(dmx, model, inp, tape=True, K=4)
    got = {}
    for mode in ("reverse", "recompute"):
        model.set_adjoint(mode)
        got[mode] = dmx.rollout_grad(out["tape"], bar, cfd=True)[0]
    a, b = got["reverse"], got["recompute"]
    assert torch.isfinite(b).all() and float((a - b).abs().max()) <= 1e-9 * float(b.abs().max())
    if B > 1:
        assert torch.equal(a[:, 1::5], bar[:, 1::5])


@pytest.mark.parametrize("call", ["grad", "grad_cfd", "params", "params_cfd"])
def test_gradients_can_be_captured(dmx, call):
    """The gradient of a tape, captured in a graph after a first call, has the bits of
    the call."""
    import torch
    B = 24
    model, inp = dmx.Model(W.toss_scene()), W.INPUTS["toss"](B, T=0.05)
    inp["x0"][:, 2] = np.where(np.arange(B) % 2 == 1, 0.055, 3.0)
    out = _call(dmx, model, inp, tape=True, K=8)
    bar = _dev(np.random.default_rng(4).normal(size=(model.nx, B)))
    fn = dmx.rollout_grad_params if call.startswith("params") else dmx.rollout_grad

    def grads():
        return [x for x in fn(out["tape"], bar, cfd=call.endswith("cfd")) if x is not None]

    want = grads()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        got = grads()
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_parameter_gradients_keep_the_order_of_their_stream(dmx):
    """The two kernels of a parameter gradient (environments with and without
    contact) start after what is queued on the call's stream, and what follows on
    it sees both results."""
    import torch
    B = 24
    model, inp = dmx.Model(W.toss_scene()), W.INPUTS["toss"](B, T=0.05)
    inp["x0"][:, 2] = np.where(np.arange(B) % 2 == 1, 0.055, 3.0)
    out = _call(dmx, model, inp, tape=True, K=8)
    bar = _dev(np.random.default_rng(4).normal(size=(model.nx, B)))
    want = [x for x in dmx.rollout_grad_params(out["tape"], bar) if x is not None]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    late = torch.zeros_like(bar)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)              # 10 ms before the cotangents are there
        late.copy_(bar)
        got = [2.0 * x for x in dmx.rollout_grad_params(out["tape"], late) if x is not None]
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, 2.0 * b)


def test_a_served_gradient_stays_within_its_admitted_memory(dmx):
    """What a gradient request takes from the device's pool while it runs is at most
    what admission counts for it (a batch whose adjoint groups are all resident,
    so that the count has no slack but its constant)."""
    _run(r'''
def high(reset=False):                          # most bytes in use at a time since the last reset (attribute 8)
    torch.cuda.synchronize()
    v = ctypes.c_uint64()
    if reset: assert rt.cudaMemPoolSetAttribute(pool, 8, ctypes.byref(v)) == 0
    assert rt.cudaMemPoolGetAttribute(pool, 8, ctypes.byref(v)) == 0
    return v.value

B = 8 * torch.cuda.get_device_properties(0).multi_processor_count
model, inp = dmx.Model(W.box_scene()), W.box_push_inputs(B, T=0.002)
req = dict(x0=np.ascontiguousarray(inp["x0"].T), T=inp["T"], grad=True, xT_bar=np.ones((13, B)), K=8, max_steps=200)
small = dmx.Server(device_bytes=1000, max_inflight=1, nstreams=1)
try:
    small.submit(model, **req)
    raise SystemExit("admitted")
except dmx.DmxError as e:
    counted = int(re.search(r"needs (\d+) device bytes", str(e)).group(1))
small.close()
srv = dmx.Server(device_bytes=8 << 30, max_inflight=1, nstreams=1)
base = used()
high(reset=True)
srv.wait(srv.submit(model, **req))
taken = high() - base
srv.close()
assert counted - (1 << 20) < taken <= counted, (taken, counted)
''')


@pytest.mark.parametrize("name", ["box", "toss", "chain_cube", "quadruped", "capsules"])
def test_cfd_parameter_gradients_match_the_oracle(dmx, orc, name):
    """Parameter gradients with contacts from distance (reverse-mode kernel: friction
    rows, capsule-box and segment pairs, box sides) against the oracle's along the
    GPU's steps, within 1e-6: moving x0 by 1e-15 moves the oracle's own by 6e-9 at
    most on these inputs."""
    from tests.test_gpu_adjoint import CFD_OPT, assert_grad, gpu_grad_params, param_inputs
    sc = W.box_scene(solref=(0.005, 1.0), **CFD_OPT) if name == "toss" else W.SCENES[name](**CFD_OPT)
    inp = (W.INPUTS["toss"](6, T=0.2) if name == "toss" else W.INPUTS[name](8) if name == "capsules" else
           param_inputs(name))
    inp.setdefault("max_steps", 20000)
    m = dmx.Model(sc)
    xT_bar = np.random.default_rng(17).normal(size=(len(inp["x0"]), m.nx))
    g = gpu_grad_params(dmx, m, inp, xT_bar, cfd=True)
    assert np.all(g["status"] == 0)
    o = orc.OracleModel(sc).batch_replay_grad(inp["x0"], inp["T"], g["hlog"], g["n"], xT_bar, ctrl=inp["ctrl"],
                                              NI=inp["NI"], cfd=True, params=True)
    assert_grad(g, o, "p_bar")
    assert_grad(g, o)


@pytest.mark.parametrize("cfd", [False, True])
def test_records_for_the_first_steps_only(dmx, cfd):
    """Segments beyond the records are recomputed: the gradient that recomputing every
    segment gives (the same right-hand sides along the same steps: 1e-12)."""
    _run(r'''
cfd = %r
model, inp = dmx.Model(W.box_scene(**(W.CFD_OPTIONS if cfd else {}))), W.box_push_inputs(64, seed=5)
bar = dev(np.random.default_rng(2).normal(size=(13, 64)))
filler = torch.empty(free() - 4 * GiB, dtype=torch.uint8, device="cuda")
got = {}
for mode in ("reverse", "recompute"):
    model.set_adjoint(mode)
    t = tape(model, inp, 0.1, K=16, rtol=1e-9, atol=1e-11, h0=1e-3)
    n, records = t.read()[1], used()
    got[mode] = dmx.rollout_grad(t, bar, cfd=cfd)[0]
    del t; gc.collect()
    assert (records > 128 << 20) == (mode == "reverse"), records
assert int(n.max()) > 288, int(n.max())         # half a GiB: at most 17 segments of 64 boxes' steps (31 KB each)
a, b = got["reverse"], got["recompute"]
assert torch.isfinite(b).all()
assert float(((a - b).abs().amax(0) / b.abs().amax(0)).max()) < 1e-12
''' % cfd)
