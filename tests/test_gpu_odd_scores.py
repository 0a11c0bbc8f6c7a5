"""Router scores that are no ordinary numbers: experts masked with -infinity and NaN.  Every choice stays a valid expert
of its own, so one such token harms no other."""
import numpy as np
import pytest
import torch

import oracle
from helpers import make_gpu_layer, make_inputs, make_oracle_layer, rel_err
from paper_2503_21135_b200 import binding
from paper_2503_21135_b200 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-2
CFG = wl.scaled(wl.CONFIGS["tiny"], top_k=3)


@pytest.fixture(scope="module")
def layer():
    wg, wu, wd, bits, pool, sets = make_inputs(CFG)
    gpu = make_gpu_layer(CFG, wg, wu, wd, bits, pool, max_tokens=700)
    ora = make_oracle_layer(CFG, wg, wu, wd, bits)
    gpu.set_channel_switch(sets)
    ora.set_channel_switch(sets)
    return gpu, ora


def _valid(idx, E):
    return idx.min() >= 0 and idx.max() < E and all(len(set(r)) == len(r) for r in idx.tolist())


@pytest.mark.parametrize("T", [7, 40, 100, 700])    # front kernel, streaming, fold and pair kernel
def test_masked_experts_are_chosen_once(layer, T):
    gpu, ora = layer
    x, lg = wl.activations(CFG, T, step=61), wl.router_logits(CFG, T, step=61)
    lg[::3, 2:] = -np.inf                            # fewer experts left than top_k
    lg[1::3, :5] = -np.inf
    y, dbg = gpu.forward(x.cuda(), lg.cuda(), binding.F32, debug=True)
    torch.cuda.synchronize()
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0
    idx, w = oracle.route(lg.numpy(), CFG.top_k)
    assert np.array_equal(dbg["idx"].cpu().numpy(), idx)
    off, perm = oracle.permute(idx, CFG.n_experts)
    assert np.array_equal(dbg["offsets"].cpu().numpy(), off) and np.array_equal(dbg["perm"].cpu().numpy(), perm)
    assert np.max(np.abs(dbg["w"].cpu().numpy() - w)) <= 1e-6
    toks = np.arange(min(T, 40), dtype=np.int32)
    ref = ora.forward(oracle.as_u16(x), lg.numpy(), tokens=toks)["y"][toks]
    assert rel_err(y.cpu().numpy()[toks], ref) <= TOL


@pytest.mark.parametrize("entry", ["logits", "router"])
@pytest.mark.parametrize("T", [7, 40, 100, 700])
def test_a_token_of_nan_scores_harms_no_other(layer, T, entry):
    gpu, _ = layer
    x, lg = wl.activations(CFG, T, step=62).cuda(), wl.router_logits(CFG, T, step=62).cuda()
    bad = [0, T // 2, T - 1]
    if entry == "router":
        w_r, bias = (t.cuda() for t in wl.router_weights(CFG))
        call = lambda x, lg: gpu.forward_router(x, w_r, bias, binding.F32, debug=True)
        x2, lg2 = x.clone(), lg
        x2[bad, 17] = float("nan")                   # one NaN input makes every score of its token NaN
    else:
        call = lambda x, lg: gpu.forward(x, lg, binding.F32, debug=True)
        x2, lg2 = x, lg.clone()
        lg2[bad] = float("nan")
        lg2[bad[1], 3] = 1.0                         # one score left
    y, dbg = call(x, lg)
    y2, dbg2 = call(x2, lg2)
    torch.cuda.synchronize()
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0
    idx = dbg2["idx"].cpu().numpy()
    assert _valid(idx, CFG.n_experts)
    good = np.setdiff1d(np.arange(T), bad)
    assert np.array_equal(idx[good], dbg["idx"].cpu().numpy()[good])
    off, perm = oracle.permute(idx, CFG.n_experts)
    assert np.array_equal(dbg2["offsets"].cpu().numpy(), off) and np.array_equal(dbg2["perm"].cpu().numpy(), perm)
    y, y2 = y.cpu().numpy(), y2.cpu().numpy()
    assert np.all(np.isnan(y2[bad]))
    assert rel_err(y2[good], y[good].astype(np.float64)) <= TOL   # an expert's rows may move to another kernel by their count
