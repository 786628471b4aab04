"""The tensor-core family on sizes it pads (AUTO's choice for bf16 models the fused family does
not take): tile edges, single columns and the largest of each range, against the oracle and
against the stepwise family that served these calls before."""
import time

import numpy as np
import pytest
import torch

import synth
from parity import check_rollout, check_teacher, np_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wm():
    import paper_2205_01435_gb300 as pkg
    return pkg.load()


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _cfg(Z, A, H, K, **flags):
    return dict(synth.model_config("small_bf16"), z_dim=Z, a_dim=A, h_dim=H, k_mix=K, **flags)


# Z, A, H, K, B, flags: one below / at / above the granularity of 8 (Z), 64 and 256 (A), 64 (H), 256 (B)
ROLLOUT = [(1, 1, 1, 1, 1, {}), (7, 63, 63, 3, 255, {}), (8, 65, 65, 8, 257, dict(ctrl_sample=1)),
           (33, 129, 130, 5, 300, dict(done_terminates=1)), (50, 257, 300, 6, 64, dict(ctrl_sample=1, value_head=1)),
           (24, 512, 128, 8, 100, dict(reward_mode=1)), (81, 200, 190, 7, 513, dict(noop_terminates=1)),
           (31, 90, 100, 4, 260, dict(n_xfers=23)), (64, 256, 512, 8, 60, {})]


@pytest.mark.parametrize("Z,A,H,K,B,flags", ROLLOUT)
def test_rollout(wm, orc, Z, A, H, K, B, flags):
    cfg, T = _cfg(Z, A, H, K, **flags), 4
    w = synth.weights(cfg, seed=31)
    z0, x = synth.z0(B, Z, seed=31), {}
    NX = cfg["n_xfers"]
    if NX:
        mask, x["loc_mask"] = synth.hier_masks(T, B, NX, A - NX, 0.5, seed=31)
    else:
        mask = synth.mask(T, B, A, 0.4, seed=31)
        mask[..., -1] |= np.uint32(0xFFFFFFFF << (A % 32) & 0xFFFFFFFF if A % 32 else 0)  # bits past A mean nothing
    if cfg["reward_mode"]:
        x["rt0"], x["mem0"] = synth.shaping_state(B, seed=31)
    h0 = np.tanh(synth.z0(B, H, seed=32)).astype(np.float32)
    c0 = synth.z0(B, H, seed=33)
    dev = {k: _cuda(v) for k, v in x.items()}
    kw = dict(h0=_cuda(h0), c0=_cuda(c0), want_seq=True, want_logp=True, **dev)  # log-probs: not the fused family
    m = wm.WorldModel(cfg, w)
    g = m.rollout(_cuda(z0), T, mask=_cuda(mask), **kw)
    m.sync()
    assert m.last_path == "tensor"
    r = check_rollout(g, cfg, w, z0, mask, h0=h0, c0=c0, orc=orc, **x)
    assert r["compared"] > 0 or B == 1
    nomask = m.rollout(_cuda(z0), T, **kw)
    assert int(nomask["actions"].max()) < (NX or A)
    # a workspace of another batch size before, and host arrays staged step by step, change nothing
    n = B // 2 + 1
    m.rollout(_cuda(z0[:n]), 2, **{k: dev[k][:n].contiguous() for k in ("rt0", "mem0") if k in dev})
    pin = {k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for k, v in dict(x, h0=h0, c0=c0).items()}
    gh = m.rollout(torch.from_numpy(z0).pin_memory(), T, mask=torch.from_numpy(mask).pin_memory(), want_seq=True,
                   want_logp=True, **pin)
    for k in ("z", "actions", "rewards", "done", "h_final", "c_final", "h_seq", "logp_seq"):
        assert torch.equal(gh[k], g[k].cpu()), k


# more gate tiles of 256 columns than 76 CTA pairs: two action rows; bf16 with a last wave half full
# (80, 114, 115, 160) and many waves; fp32 on both sides of its rule (40, 316, 320, 330, 512)
@pytest.mark.parametrize("H,B,precision,NX", [
    (256, 9985, "bf16", 32), (512, 5001, "bf16", 32), (512, 2500, "bf16", 0), (1216, 1281, "bf16", 0),
    (320, 5800, "bf16", 0), (1024, 2500, "bf16", 0), (512, 40001, "bf16", 0), (512, 1100, "fp32", 0), (256, 20001, "fp32", 0),
    (512, 10200, "fp32", 0), (704, 7600, "fp32", 0), (512, 16300, "fp32", 0)])
def test_gates_over_many_tiles(wm, H, B, precision, NX):
    """The bits of the same episodes in a batch of few tiles (which the oracle checks)."""
    cfg, T = dict(_cfg(32, 128, H, 5, ctrl_sample=1, n_xfers=NX), precision=precision), 3
    z0, x = synth.z0(B, 32, seed=35), {}
    if NX:
        x["mask"], x["loc_mask"] = synth.hier_masks(T, B, NX, 128 - NX, 0.5, seed=35)
    m = wm.WorldModel(cfg, synth.weights(cfg, seed=35))
    g = m.rollout(_cuda(z0), T, want_seq=True, want_logp=True, **{k: _cuda(v) for k, v in x.items()})
    for first in (0, B - 300):
        r = slice(first, first + 300)
        s = m.rollout(_cuda(z0[r]), T, episode_offset=first, want_seq=True, want_logp=True,
                      **{k: _cuda(v[:, r]) for k, v in x.items()})
        assert m.last_path == "tensor"
        for k in ("z", "h_seq", "rewards"):
            assert torch.equal(s[k], g[k][:, r]), k
        assert torch.equal(s["c_final"], g["c_final"][r])


@pytest.mark.parametrize("Z,A,H,K,N,T", [(5, 45, 333, 3, 700, 3), (50, 101, 300, 6, 600, 5), (64, 256, 512, 5, 60, 4)])
def test_scoring_and_training(wm, orc, Z, A, H, K, N, T):
    cfg = _cfg(Z, A, H, K)
    w = synth.weights(cfg, seed=34)
    zs, acts, lens = synth.teacher_inputs(N, T, Z, A, seed=34, ragged=True)
    acts[::2, ::3] = -1
    m = wm.WorldModel(cfg, w)
    g = m.mdn_nll(_cuda(zs), _cuda(acts), lengths=_cuda(lens), want_seq=True)
    m.sync()
    assert m.last_path == "tensor"
    check_teacher({k: np_(v) for k, v in g.items()}, orc.mdn_nll(cfg, w, zs, acts, lengths=lens, want_seq=True), "bf16")
    a = m.mdn_nll_backward(_cuda(zs), _cuda(acts), lengths=_cuda(lens))
    s = wm.WorldModel(dict(cfg, path="stepwise"), w).mdn_nll_backward(_cuda(zs), _cuda(acts), lengths=_cuda(lens))
    for k in ("W_lstm", "b_lstm", "W_mdn", "b_mdn", "nll"):
        # both forwards round the same operands to bf16 (2^-9 each) and sum in fp32
        assert float((a[k] - s[k]).norm() / s[k].norm()) < 1e-2, k


def test_forced_path_still_refuses_unaligned_sizes(wm):
    cfg = _cfg(50, 101, 300, 6, path="tensor")
    m = wm.WorldModel(cfg, synth.weights(cfg))
    with pytest.raises(wm.WMError) as e:
        m.rollout(torch.zeros(300, 50, device="cuda"), 1)
    assert e.value.status == wm.WM_ERR_UNSUPPORTED


@pytest.mark.parametrize("Z,A,H,K,B,flags", [(50, 101, 300, 6, 40, {}), (31, 90, 100, 4, 260, dict(n_xfers=23)),
                                             (33, 129, 130, 5, 300, dict(done_terminates=1))])
def test_infinite_latents_stay_in_their_row_and_step(wm, Z, A, H, K, B, flags):
    """An infinite latent saturates the gates it meets; the padded units, whose weights are 0, make no NaN of it."""
    cfg, T = _cfg(Z, A, H, K, **flags), 3
    w = synth.weights(cfg, seed=39)
    z0, x = synth.z0(B, Z, seed=39), {}
    z0[0, 3], z0[1, 2], z0[B - 1, Z - 1] = np.inf, -np.inf, 3.4e38  # (the last rounds to infinity in bf16)
    NX = cfg["n_xfers"]
    if NX:
        mask, x["loc_mask"] = (_cuda(v) for v in synth.hier_masks(T, B, NX, A - NX, 0.5, seed=39))
    else:
        mask = _cuda(synth.mask(T, B, A, 0.4, seed=39))
    g, s = (wm.WorldModel(dict(cfg, path=p), w).rollout(_cuda(z0), T, mask=mask, want_logp=True, want_seq=True, **x)
            for p in ("auto", "stepwise"))
    same = (g["actions"] == s["actions"]).all(0) & (g["comp_seq"] == s["comp_seq"]).all(2).all(0)
    assert same[[0, 1, B - 1]].any()
    for k in ("h_seq", "c_seq", "rewards", "mdn_seq"):
        assert torch.isfinite(g[k]).all(), k
        assert float((g[k][:, same] - s[k][:, same]).abs().max()) < 2e-2, k  # (the parity bound of bf16 paths)


@pytest.mark.parametrize("Z,A,H,K,N,T", [(50, 101, 300, 6, 40, 12), (11, 45, 100, 3, 200, 11)])
def test_infinite_targets_past_a_sequence_do_not_spread(wm, Z, A, H, K, N, T):
    cfg = _cfg(Z, A, H, K)
    w = synth.weights(cfg, seed=40)
    zs, acts, _ = synth.teacher_inputs(N, T, Z, A, seed=40)
    zs[5, ::3, 1] = np.inf
    lens = np.full(N, 4, np.int32)
    m = wm.WorldModel(cfg, w)
    g = m.mdn_nll(_cuda(zs), _cuda(acts), lengths=_cuda(lens), want_seq=True)
    assert m.last_path == "tensor"
    s = wm.WorldModel(dict(cfg, path="stepwise"), w).mdn_nll(_cuda(zs), _cuda(acts), lengths=_cuda(lens), want_seq=True)
    for k in g:
        assert torch.isfinite(g[k]).all(), k
        assert float((g[k] - s[k]).norm() / s[k].norm()) < 1e-2, k


# sizes padded, and a small batch of an aligned model; a second action row
ACCURATE = [(50, 101, 300, 6, 300, 0), (64, 256, 512, 8, 60, 0), (31, 90, 100, 4, 260, 23), (24, 512, 128, 8, 100, 0)]


@pytest.mark.parametrize("Z,A,H,K,B,NX", ACCURATE)
def test_small_sigmoids_keep_their_relative_accuracy(wm, Z, A, H, K, B, NX):
    """Zero weights, gate biases i = o = -18, f = -30, g = 1: c' = sigma(-18) tanh(1), h' = sigma(-18) tanh(c')."""
    cfg = _cfg(Z, A, H, K, n_xfers=NX)
    w = {k: np.zeros_like(v) if isinstance(v, np.ndarray) else v for k, v in synth.weights(cfg, seed=1).items()}
    w["b_lstm"] = np.repeat(np.float32([-18, -30, 1, -18]), H)
    s18 = 1 / (1 + np.exp(18.0))
    c = s18 * np.tanh(1.0)
    m = wm.WorldModel(cfg, w)
    outs = [m.rollout(torch.zeros(B, Z, device="cuda"), 1, want_seq=True, want_logp=True)]
    assert m.last_path == "tensor"
    if not NX:
        for T in (1, 12):  # one launch per step (a fused member at H = 128), and one launch
            outs.append(m.mdn_nll(torch.zeros(T + 1, B, Z, device="cuda"),
                                  torch.full((T, B), -1, dtype=torch.int32, device="cuda"), want_seq=True))
            assert m.last_path == ("fused" if T == 1 and H == 128 else "tensor")
            if m.last_path == "fused":
                outs.pop()  # (its exponential is the hardware's)
    for g in outs:
        # expf, tanhf (2 ulp each), an addition, a reciprocal, a product: under 16 fp32 roundoffs
        np.testing.assert_allclose(np_(g["c_seq"][0]), c, rtol=16 * 2.0**-24)
        np.testing.assert_allclose(np_(g["h_seq"][0]), s18 * np.tanh(c), rtol=24 * 2.0**-24)


@pytest.mark.parametrize("Z,A,H,K,B,NX", [v for v in ACCURATE if not v[-1]])
def test_draws_weigh_logits_accurately(wm, Z, A, H, K, B, NX):
    """Logits that are the bias alone, large beside their differences: the log-probability of the drawn
    action against 64 bits."""
    cfg = _cfg(Z, A, H, K, ctrl_sample=1, ctrl_tau=0.05)
    w = synth.weights(cfg, seed=2)
    w["W_ctrl"] = np.zeros_like(w["W_ctrl"])
    w["b_ctrl"] = (100 + np.random.default_rng(2).random(A) * 0.5).astype(np.float32)
    mask = synth.mask(1, B, A, 0.5, seed=2)
    m = wm.WorldModel(cfg, w)
    g = m.rollout(_cuda(synth.z0(B, Z, seed=2)), 1, mask=_cuda(mask), want_logp=True)
    assert m.last_path == "tensor"
    acts = np_(g["actions"])[0]
    valid = np.unpackbits(mask[0].view(np.uint8), axis=-1, bitorder="little")[:, :A].astype(bool)
    l = np.where(valid, w["b_ctrl"].astype(np.float64) / np.float64(np.float32(0.05)), -np.inf)
    top = l.max(-1, keepdims=True)
    lp = l - top - np.log(np.exp(l - top).sum(-1, keepdims=True))
    ok = acts >= 0
    assert ok.sum() > B // 2
    # a quotient up to 10 (2^-24 of it), exponentials (2 ulp each), their sum and its logarithm
    np.testing.assert_allclose(np_(g["logp_seq"])[0][ok], lp[np.arange(B), acts][ok], rtol=0, atol=64 * 2.0**-24)


def _scoring(N, T, Z, A):
    g = torch.Generator(device="cuda").manual_seed(3)
    return (torch.randn((T + 1, N, Z), generator=g, device="cuda"),
            torch.randint(0, A, (T, N), generator=g, device="cuda", dtype=torch.int32))


@pytest.mark.parametrize("train", [False, True])
def test_a_longer_call_is_captured_after_a_short_one(wm, train):
    """The operand rows of more steps would have to be allocated under capture: the call goes to the family
    whose scratch does not grow with the steps.  (A training step's own workspace grows with the rows: a
    call of more rows comes first.)"""
    cfg = _cfg(50, 101, 300, 6)
    w = synth.weights(cfg, seed=36)
    m = wm.WorldModel(cfg, w)
    z, a = _scoring(70, 24, 50, 101)
    run = m.mdn_nll_backward if train else m.mdn_nll
    run(z[:5], a[:4])  # (the operand rows of 4 steps)
    if train:
        run(*_scoring(100, 24, 50, 101))
    m.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = run(z, a)
    path = m.last_path
    for v in got.values():
        v.zero_()
    g.replay()
    torch.cuda.synchronize()
    if not train:
        assert path == "stepwise"
    want = (lambda s: s.mdn_nll_backward(z, a) if train else s.mdn_nll(z, a))(wm.WorldModel(cfg, w))
    for k in want:  # bf16 operands on both families, sums in another order
        assert float((got[k] - want[k]).norm() / want[k].norm()) < (5e-3 if train else 1e-5), k


def test_a_call_whose_operand_rows_have_no_room(wm):
    """Scoring that the tensor family would need 4 GB for runs on N rows' scratch when 2 GB are free."""
    N, T, cfg = 12000, 400, _cfg(50, 101, 300, 6)
    m = wm.WorldModel(cfg, synth.weights(cfg, seed=37))
    z, a = _scoring(N, T, 50, 101)
    m.mdn_nll(z[:2, :, :], a[:1])
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    got = m.mdn_nll(z, a)["nll"]
    m.sync()
    assert m.last_path == "stepwise"
    del hold
    torch.cuda.empty_cache()
    want = m.mdn_nll(z, a)["nll"]
    m.sync()
    assert m.last_path == "tensor"
    assert float((got - want).norm() / want.norm()) < 1e-5


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_training_step_holds_what_it_reads(wm, prec):
    """Device memory of a first training step: the buffers of the batched backward, with an eighth to spare."""
    Z, A, H, K, N, T = 64, 256, 512, 5, 512, 64
    cfg = dict(_cfg(Z, A, H, K), precision=prec)
    m = wm.WorldModel(cfg, synth.weights(cfg, seed=38))
    z, a = _scoring(N, T, Z, A)
    m.mdn_nll_backward(z[:3], a[:2])  # the libraries' own memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    r0 = torch.cuda.memory_reserved()
    m.mdn_nll_backward(z, a)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0] - (torch.cuda.memory_reserved() - r0)
    M, b = 3 * K * Z, prec == "bf16"
    rows = 4 * (H + 4 * H + M + H + 4 * H) + (2 * (M + 4 * H) if b else 4 * H)  # c, G, dMD, dY, dG (and copies, or h)
    rows += (2 if b else 4) * (Z + H) + 4 * 4 * 8                                 # frames, the likelihood's partials
    assert used < 1.125 * N * T * rows + (96 << 20), (used, N * T * rows)


def test_pageable_outputs_do_not_hold_up_the_steps(wm):
    """A call with every output in pageable host memory takes no longer than on the family whose host arrays
    are copied whole (copied step by step it took seven times as long)."""
    Z, A, H, K, B, T = 50, 101, 300, 6, 2000, 30
    cfg = _cfg(Z, A, H, K)
    w, z0 = synth.weights(cfg, seed=46), torch.from_numpy(synth.z0(B, Z, seed=46))
    mask = torch.from_numpy(synth.mask(T, B, A, 0.4, seed=46))

    def best(path):
        m, ms = wm.WorldModel(dict(cfg, path=path), w), []
        m.rollout(z0, T, mask=mask, want_seq=True)
        for _ in range(4):
            t = time.perf_counter()
            m.rollout(z0, T, mask=mask, want_seq=True)  # (allocates its outputs)
            ms.append(time.perf_counter() - t)
        return min(ms), m.last_path

    (auto, path), (step, _) = best("auto"), best("stepwise")
    assert path == "tensor" and auto < 1.5 * step, (auto, step)
