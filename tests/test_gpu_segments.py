"""The passes that find their trajectories by searching cu_seqlens (advantages
with gamma = lambda = 1, with a fixed and with a length-adaptive lambda,
step-level advantages, the clipped surrogate's counts, the GRPO and running-mean
broadcasts) on layouts
where the search can go wrong: one trajectory, runs of empty ones at the chunk
edges, more than 32 and more than 1,024 of them inside one chunk, ends exactly
on chunk edges, and batches on both sides of the sizes at which the group and
running-mean passes look at the batch differently. Bars as in those passes' own
tests."""
import numpy as np
import pytest
import torch

from oracle import sao_oracle as O
from paper_2607_07508_gb300 import sao, synthetic as S
from tests._util import cuda, rel_err_floor

pytestmark = pytest.mark.gpu

LAYOUTS = [[1], [1024], [5000], [1024, 1024, 1], [0] * 40 + [1024] + [0] * 70 + [1023, 1, 0, 2048],
           [1] * 1500 + [3000], [16384, 0, 16383, 1, 32768, 5], [7, 0, 3] * 900 + [9000] + [0] * 33, [8192, 0, 8192, 16384], [16] * 2050]


def f32(x):
    return float(np.float32(x))


@pytest.mark.parametrize("k", range(len(LAYOUTS)))
def test_segment_passes(k):
    wl = S.make_custom(LAYOUTS[k], 8, 16, "f32", seed=100 + k, dense=False, obs_frac=0.4)
    N, B = wl.N, wl.B
    rng = np.random.default_rng(k)
    v, m, cu, rew = cuda(wl.values), cuda(wl.loss_mask), cuda(wl.cu_seqlens), cuda(wl.rewards)
    ws = sao.workspace(N)
    nan = lambda: torch.full((N,), float("nan"), device="cuda")
    for lam, alpha in ((1.0, 0.0), (f32(0.95), 0.0), (1.0, 1.5)):
        adv, ret = nan(), nan()
        sao.sao_advantages(v, rew, m, cu, 1.0, lam, 1.0, alpha, adv, ret, ws)
        wa, wr = O.advantages(wl.values, wl.rewards, wl.loss_mask, wl.cu_seqlens, 1.0, lam, 1.0, alpha)
        assert rel_err_floor(adv.cpu().numpy(), wa, 1e-3).max() <= 1e-5
        assert rel_err_floor(ret.cpu().numpy(), wr, 1e-3).max() <= 1e-5
    for mode in (sao.SAO_STEP_AVERAGE, sao.SAO_STEP_LAST):
        adv, ret, vm = nan(), nan(), torch.full((N,), 9, dtype=torch.uint8, device="cuda")
        sao.sao_step_advantages(v, rew, m, cu, 1.0, f32(0.95), 1.0, 0.0, mode, adv, ret, ws, value_mask=vm)
        wa, wr, wv = O.step_advantages(wl.values, wl.rewards, wl.loss_mask, wl.cu_seqlens, 1.0, f32(0.95), 1.0, 0.0,
                                       mode)
        assert rel_err_floor(adv.cpu().numpy(), wa, 1e-3).max() <= 1e-5
        assert rel_err_floor(ret.cpu().numpy(), wr, 1e-3).max() <= 1e-5
        assert np.array_equal(vm.cpu().numpy(), wv)
    logp = (-rng.exponential(2.0, N)).astype(np.float32)
    old = (logp + rng.normal(0, 0.2, N)).astype(np.float32)
    a = rng.normal(size=N).astype(np.float32)
    loss, counts = torch.empty(1, device="cuda"), torch.empty(4, dtype=torch.int64, device="cuda")
    for norm in (sao.SAO_NORM_TOKEN, sao.SAO_NORM_SEQUENCE):
        coef, grad = nan(), nan()
        args = (cuda(logp), cuda(old), cuda(a), m, cu, 0.2, 0.28, norm)
        sao.sao_clip_loss_fwd(*args, loss, counts, ws, coef=coef)
        sao.sao_clip_loss_bwd(*args, torch.ones(1, device="cuda"), grad, ws)
        want = O.clip_loss(logp, old, a, wl.loss_mask, wl.cu_seqlens, 0.2, 0.28, norm)
        assert abs(loss.item() - want["loss"]) <= 1e-4 * max(abs(want["loss"]), 1e-6)
        assert rel_err_floor(coef.cpu().numpy(), want["coef"], 1e-12).max() <= 1e-5
        assert torch.equal(coef, grad)
        assert counts[0].item() == int(wl.loss_mask.sum())
    for gid in (np.arange(B) // 4, rng.permutation(np.arange(B) // 4)):
        adv = nan()
        gid = gid.astype(np.int32)
        sao.sao_group_advantages(rew, cuda(gid), m, cu, f32(1e-6), adv, ws)
        want = O.group_advantages(wl.rewards, gid, wl.loss_mask, wl.cu_seqlens, f32(1e-6))
        assert rel_err_floor(adv.cpu().numpy(), want, 1e-3).max() <= 1e-5
    for P, window in ((3, 8), (97, 4)):
        pid = rng.integers(0, P, B).astype(np.int32)
        hist = rng.random((P, window)).astype(np.float32)
        seen = rng.integers(0, 3 * window, P).astype(np.int64)
        th, ts, adv = cuda(hist), cuda(seen), nan()
        sao.sao_running_mean_advantages(rew, cuda(pid), th, ts, m, cu, adv, ws)
        want, wh, wseen = O.running_mean_advantages(wl.rewards, pid, wl.loss_mask, wl.cu_seqlens, hist, seen, window)
        assert rel_err_floor(adv.cpu().numpy(), want, 1e-3).max() <= 1e-5
        assert np.array_equal(ts.cpu().numpy(), wseen) and np.allclose(th.cpu().numpy(), wh)


def test_telescoped_call_checks_cu_seqlens():
    v = torch.zeros(30, device="cuda")
    m = torch.ones(30, dtype=torch.uint8, device="cuda")
    adv, ret, ws = torch.empty_like(v), torch.empty_like(v), sao.workspace(30)
    sao.sao_set_checked(True)
    try:
        for bad in ([0, 20, 15, 30], [1, 20, 30], [0, 20, 29]):
            cu = torch.tensor(bad, dtype=torch.int32, device="cuda")
            with pytest.raises(sao.SaoError) as e:
                sao.sao_advantages(v, torch.zeros(len(bad) - 1, device="cuda"), m, cu, 1.0, 1.0, 1.0, 0.0, adv, ret, ws)
            assert e.value.status == 6
    finally:
        sao.sao_set_checked(False)


@pytest.mark.parametrize("layout", [[3] * 1024, [3] * 1025, [2] * 2048, [2] * 2049, [2, 0, 1] * 4097,
                                    [260000, 0, 270000, 260000], [700] * 1025 + [90000]],
                         ids=["1024", "1025", "2048", "2049", "12291", "more than a wave", "1026, more than a wave"])
def test_clip_totals(layout):
    """The clipped surrogate's totals added by each CTA (up to 1,024 trajectories)
    and by a launch of 2,048 trajectories per CTA, with the loss added by its last CTA
    and by a launch of its own. Bars as in test_segment_passes; trajectories without an action token."""
    rng = np.random.default_rng(len(layout))
    cu = np.concatenate([[0], np.cumsum(layout)]).astype(np.int32)
    N = int(cu[-1])
    m = (rng.random(N) < 0.6).astype(np.uint8)
    m[cu[1]:cu[2]] = 0
    logp = (-rng.exponential(2.0, N)).astype(np.float32)
    old = (logp + rng.normal(0, 0.2, N)).astype(np.float32)
    a = rng.normal(size=N).astype(np.float32)
    loss, counts, ws = torch.empty(1, device="cuda"), torch.empty(4, dtype=torch.int64, device="cuda"), sao.workspace(N)
    for norm in (sao.SAO_NORM_TOKEN, sao.SAO_NORM_SEQUENCE):
        coef, grad = torch.full((N,), float("nan"), device="cuda"), torch.full((N,), float("nan"), device="cuda")
        args = (cuda(logp), cuda(old), cuda(a), cuda(m), cuda(cu), 0.2, 0.28, norm)
        sao.sao_clip_loss_fwd(*args, loss, counts, ws, coef=coef)
        sao.sao_clip_loss_bwd(*args, torch.ones(1, device="cuda"), grad, ws)
        want = O.clip_loss(logp, old, a, m, cu, 0.2, 0.28, norm)
        # weighted terms of both signs: against the sum of their magnitudes
        scale = float(np.abs(want["coef"]).sum())
        assert abs(loss.item() - want["loss"]) <= 1e-6 * max(scale, abs(want["loss"]))
        assert rel_err_floor(coef.cpu().numpy(), want["coef"], 1e-12).max() <= 1e-5
        assert torch.equal(coef, grad)
        assert counts[0].item() == int(m.sum())
