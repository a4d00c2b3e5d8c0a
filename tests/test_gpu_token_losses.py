"""The per-token losses on both sides of the size where one cluster stops doing
the whole call (32,768 tokens), with ragged ends, arrays one element off
16-byte alignment, and the normaliser counted or given; bars as in the tests of
each loss (fp32 products, sums in more than fp32)."""
import numpy as np
import pytest
import torch

from tests.test_gpu_next import _check_decoupled
from tests.test_gpu_on_kernels import _check_pl, _vl_gpu
from oracle import sao_oracle as O
from paper_2607_07508_gb300 import sao
from tests._util import rel_err_floor

pytestmark = pytest.mark.gpu


def _inputs(N):
    rng = np.random.default_rng(N)
    logp = (-rng.exponential(2.0, N)).astype(np.float32)
    old = (logp + rng.normal(0, 0.3, N)).astype(np.float32)
    roll = (old + rng.normal(0, 0.4, N)).astype(np.float32)
    adv = rng.normal(size=N).astype(np.float32)
    mask = (rng.random(N) < 0.7).astype(np.uint8)
    return logp, old, roll, adv, mask


@pytest.mark.parametrize("N", [2, 4096, 4097, 8191, 32767, 32768, 32769, 32772, 65535, 65536, 65537, 65540, 131073, 400003])
def test_token_losses_at_the_cluster_line(N):
    logp, old, roll, adv, mask = _inputs(N)
    for offset in (0, 1):
        _check_pl(logp, old, adv, mask, 0.3, 5.0, offset=offset)
        _check_pl(logp, old, adv, mask, 0.8, 3.0, n_norm=2 * N + 1, offset=offset)
    _check_decoupled(logp, old, roll, adv, mask, 0.2, 0.28, 0.5, 2.0)
    _check_decoupled(logp, old, roll, adv, mask, 0.2, 0.28, 0.5, 2.0, n_norm=777)
    _check_vl(logp, adv, mask)


def _check_vl(values, ret, mask):
    N = len(values)
    for n_norm in (0, 3 * N):
        loss, grad, ev = _vl_gpu(values, ret, mask, n_norm)
        wl, wg, wev = O.value_loss(values, ret, mask, n_norm)
        assert abs(loss - wl) <= 1e-4 * abs(wl)
        assert rel_err_floor(grad, wg, 1e-12).max() <= 1e-5
        assert np.allclose(ev, wev, rtol=1e-9, atol=1e-9 * np.abs(wev).max())


@pytest.mark.parametrize("N", [1 << 18, (1 << 18) + 1025, 1 << 20, (1 << 20) + 5])
def test_value_loss_at_the_narrow_grid_line(N):
    """One CTA per SM from more than 256 CTAs' worth of tokens up to 2^20 of them, a full wave above."""
    logp, _, _, adv, mask = _inputs(N)
    _check_vl(logp, adv, mask)


@pytest.mark.parametrize("N", [20000, 100000, 1 << 19])
def test_sums_beyond_fp32_range(N):
    """Sums of squares above 3.4e38, and of terms above it, are fp64 sums: finite."""
    logp, old, roll, adv, mask = _inputs(N)
    _check_vl(logp, adv * np.float32(1e17), mask)
    adv = np.full(N, 2e37, np.float32)  # four tokens' terms stay below 3.4e38
    _check_pl(logp, old, adv, mask, 0.3, 1.0)
    _check_decoupled(logp, old, roll, adv, mask, 0.2, 0.28, 0.5, 2.0)


@pytest.mark.parametrize("N", [20000, 100000])
def test_ev_sums_keep_53_bits(N):
    """Squares of three sizes, one to a thread, whose sum is a whole number below 2^53: exact."""
    ret = np.zeros(N, np.float32)
    ret[::4] = 1.0
    ret[::64] = 2.0 ** 13
    ret[4 * 777] = 2.0 ** 26
    zero, ones = np.zeros(N, np.float32), np.ones(N, np.uint8)
    _, _, ev = _vl_gpu(zero, ret, ones, 0)
    want = int((ret.astype(np.int64) ** 2).sum())
    assert want < 1 << 53 and int(ev[1]) == want and int(ev[3]) == want


@pytest.mark.parametrize("N", [1000, 70000])
def test_ev_sums_of_the_smallest_numbers(N):
    """Multiples of fp32's smallest number add up exactly in fp64."""
    k = 2 * np.random.default_rng(N).integers(0, 1000, N) + 1
    ret = np.ldexp(k.astype(np.float64), -149).astype(np.float32)
    _, _, ev = _vl_gpu(np.zeros(N, np.float32), ret, np.ones(N, np.uint8), 0)
    assert ev[2] == ev[0] == np.ldexp(float(k.sum()), -149)


@pytest.mark.parametrize("N", [1, 3, 17, 35, 1001, 32769, 70003])
def test_action_counts_at_every_mask_alignment(N):
    g = torch.Generator(device="cuda").manual_seed(N)
    mask = (torch.rand(N, generator=g, device="cuda") < 0.6).to(torch.uint8) * 7
    zeros, one = torch.zeros(N, device="cuda"), torch.ones(N, device="cuda")
    ws, loss = sao.workspace(N), torch.empty(1, device="cuda")
    counts, grad = torch.empty(4, dtype=torch.int64, device="cuda"), torch.empty(N, device="cuda")
    n = int((mask != 0).sum())
    for offset in range(16):
        m = torch.full((N + 32,), 255, dtype=torch.uint8, device="cuda")[offset:offset + N].copy_(mask)
        sao.sao_policy_loss_fwd(zeros, zeros, one, m, 0.2, 0.28, loss, counts, ws)
        sao.sao_value_loss(one, zeros, m, loss, grad, ws)
        assert counts.tolist() == [n, 0, 0, 0] and float(loss) == (1.0 if n else 0.0)
