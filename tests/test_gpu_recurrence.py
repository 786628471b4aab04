"""The one-launch teacher-forced recurrence: row-tile edges (128), clusters and unit tiles of every
hidden size it splits, several row tiles per CTA, rings shorter than a tile's operands, against the
oracle; determinism; and the calls it leaves to one launch per step."""
import numpy as np
import pytest
import torch

import synth
from parity import check_teacher, np_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wm():
    import paper_2205_01435_gb300 as pkg
    return pkg.load()


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# Z, A, H, K, N, T, precision (aligned sizes: the tensor family takes both precisions), one launch or one per step
# (more row tiles than four per CTA; weights that do not fit)
CASES = [(8, 64, 64, 2, 300, 5, "bf16", True), (64, 64, 64, 5, 1, 4, "fp32", True), (24, 128, 320, 5, 129, 6, "bf16", True),
         (64, 256, 512, 5, 127, 3, "fp32", True), (64, 256, 512, 5, 257, 4, "bf16", True), (64, 256, 512, 5, 1000, 4, "bf16", True),
         (64, 256, 512, 5, 640, 3, "fp32", True), (128, 512, 1024, 8, 256, 3, "bf16", True), (128, 512, 1024, 8, 300, 2, "bf16", True),
         (32, 64, 256, 5, 2500, 3, "bf16", True), (32, 64, 256, 5, 9800, 2, "bf16", False), (128, 512, 1024, 8, 40, 2, "fp32", False)]


@pytest.mark.parametrize("Z,A,H,K,N,T,prec,one", CASES)
def test_scoring_against_oracle(wm, orc, Z, A, H, K, N, T, prec, one):
    cfg = dict(synth.model_config("nll"), z_dim=Z, a_dim=A, h_dim=H, k_mix=K, precision=prec)
    w = synth.weights(cfg, seed=41)
    zs, acts, lens = synth.teacher_inputs(N, T, Z, A, seed=41, ragged=True)
    acts[1::2, ::5] = -1
    m = wm.WorldModel(dict(cfg, path="tensor"), w)
    args = (_cuda(zs), _cuda(acts))
    g = m.mdn_nll(*args, lengths=_cuda(lens), want_seq=True)
    m.sync()
    assert m.last_launches == 4 + (1 if one else T)  # the state, the frames, the recurrence, the heads, the sums
    idx = np.unique(np.linspace(0, N - 1, 24).round().astype(int))
    o = orc.mdn_nll(cfg, w, zs[:, idx], acts[:, idx], lengths=lens[idx], want_seq=True)
    check_teacher({k: np_(v)[idx] if k == "nll" else np_(v)[:, idx] for k, v in g.items()}, o, prec)
    again = m.mdn_nll(*args, lengths=_cuda(lens), want_seq=True)
    plain = m.mdn_nll(*args, lengths=_cuda(lens))  # the other outputs change nothing
    for k in g:
        assert torch.equal(g[k], again[k]), k
    assert torch.equal(g["nll"], plain["nll"])
    # a sequence's likelihood does not depend on the batch around it
    one = m.mdn_nll(_cuda(zs[:, N - 1:]), _cuda(acts[:, N - 1:]), lengths=_cuda(lens[N - 1:]), want_seq=True)
    assert torch.equal(one["h_seq"][:, 0], g["h_seq"][:, N - 1])


def test_bad_action_on_the_device_is_reported(wm):
    cfg = synth.model_config("nll")
    m = wm.WorldModel(dict(cfg, path="tensor"), synth.weights(cfg))
    zs, acts, _ = synth.teacher_inputs(200, 4, 64, 256, seed=42)
    acts[2, 150] = 256
    m.mdn_nll(_cuda(zs), _cuda(acts))
    with pytest.raises(wm.WMError) as e:
        m.sync()
    assert e.value.status == wm.WM_ERR_INVALID_ARG


def test_under_stream_capture(wm):
    """A captured call replays to the same bits."""
    cfg = synth.model_config("nll")
    m = wm.WorldModel(dict(cfg, path="tensor"), synth.weights(cfg))
    zs, acts, _ = synth.teacher_inputs(300, 6, 64, 256, seed=43)
    z, a = _cuda(zs), _cuda(acts)
    want = m.mdn_nll(z, a, want_seq=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = m.mdn_nll(z, a, want_seq=True)
    for k in got:
        got[k].zero_()
    g.replay()
    torch.cuda.synchronize()
    for k in want:
        assert torch.equal(want[k], got[k]), k


# the backward recurrence: cluster edges of every hidden size (64 units), row-tile edges, two launches
# (more row tiles than the SMs hold), one step (no recurrence), the fp32 parts, sizes it leaves.
# Launches: the forward's (1 on a fused member, 5 on the tensor family with one recurrence launch), before the
# recurrence (dY; with a forward that leaves nothing also the operands, the gates' GEMM and kernel and the mixture's
# gradient), the recurrence (2 T - 1 step by step), and 3 GEMMs and 7 sums
BACKWARD = [(8, 64, 64, 3, 129, 3, "bf16", 1 + 5 + 1 + 10), (16, 64, 64, 2, 1, 2, "fp32", 1 + 5 + 1 + 10),
            (64, 256, 512, 5, 130, 4, "bf16", 5 + 1 + 1 + 10), (64, 256, 512, 5, 200, 3, "fp32", 5 + 1 + 1 + 10),
            (16, 64, 512, 2, 700, 3, "bf16", 5 + 1 + 2 + 10), (16, 64, 512, 2, 600, 2, "fp32", 5 + 1 + 2 + 10),
            (32, 128, 1024, 3, 140, 2, "bf16", 5 + 1 + 1 + 10), (16, 64, 1024, 2, 20, 2, "fp32", 6 + 4 + 3 + 10),
            (24, 128, 320, 5, 60, 4, "bf16", 5 + 1 + 1 + 10), (16, 64, 128, 2, 50, 1, "bf16", 1 + 5 + 1 + 10),
            (11, 45, 100, 3, 40, 5, "bf16", 1 + 5 + 9 + 10)]


@pytest.mark.parametrize("Z,A,H,K,N,T,prec,launches", BACKWARD)
def test_gradient_against_oracle(wm, orc, Z, A, H, K, N, T, prec, launches):
    cfg = dict(synth.model_config("nll"), z_dim=Z, a_dim=A, h_dim=H, k_mix=K, precision=prec)
    w = synth.weights(cfg, seed=44)
    zs, acts, lens = synth.teacher_inputs(N, T, Z, A, seed=44, ragged=True)
    acts[1::2, ::5] = -1
    m = wm.WorldModel(cfg, w)
    args = (_cuda(zs), _cuda(acts), _cuda(lens))
    g = m.mdn_nll_backward(*args)
    m.sync()
    assert m.last_launches == launches
    o = orc.mdn_nll_grad(cfg, w, zs, acts, lens, nthreads=16)
    # relative Frobenius norms: about 100 fp32 roundoffs, 4 bf16 roundoffs (the operands are rounded once)
    tol = {"fp32": 1e-5, "bf16": 1e-2}[prec]
    for k in ("W_lstm", "b_lstm", "W_mdn", "b_mdn"):
        ref = np.asarray(o[k], np.float64)
        assert np.linalg.norm(np_(g[k]) - ref) <= tol * max(np.linalg.norm(ref), 1e-30), k
    again = m.mdn_nll_backward(*args)
    for k in g:
        assert torch.equal(g[k], again[k]), k


def test_launches_are_counted(wm):
    """fp32, H = 1024: one gate GEMM per step, the head GEMM forms the gradient, and the backward goes step by
    step: operands, gates (GEMM and kernel), dY; a cell kernel a step and a GEMM between; 3 GEMMs; 7 sums."""
    cfg, T = dict(synth.model_config("nll"), z_dim=16, a_dim=64, h_dim=1024, k_mix=2, precision="fp32"), 3
    zs, acts, _ = synth.teacher_inputs(20, T, 16, 64, seed=45)
    m = wm.WorldModel(cfg, synth.weights(cfg, seed=45))
    m.mdn_nll(_cuda(zs), _cuda(acts))
    assert m.last_path == "tensor" and m.last_launches == 4 + T
    m.mdn_nll_backward(_cuda(zs), _cuda(acts))
    assert m.last_launches == 4 + T + 4 + (2 * T - 1) + 3 + 7
