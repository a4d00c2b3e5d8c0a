"""bf16 log-prob backward on few rows: the dH product cut along the vocabulary,
and dW through staged boxes or one M tile per CTA tile, written or added to, at
the edges of the 128-row / 32-column boxes and of the token ranges that choose
between them. Against fp64 (torch), with bf16 dZ and dH roundings (2^-9 each,
random) inside 1e-2 in the 2-norm."""
import pytest
import torch

from paper_2607_07508_gb300 import sao

pytestmark = pytest.mark.gpu

TOL = 1e-2


def _rel(got, want):
    return float((got.double() - want).norm() / want.norm().clamp(min=1e-300))


@pytest.mark.parametrize("N,h,V", [(1, 8, 300), (129, 40, 1153), (517, 1000, 2049), (1279, 264, 999),
                                   (1280, 264, 999), (3071, 72, 640), (3072, 72, 640), (40, 136, 70000)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_backward_few_rows(N, h, V, accumulate):
    g = torch.Generator(device="cuda").manual_seed(N + h)
    H = torch.randn(N, h, generator=g, device="cuda").bfloat16()
    W = (torch.randn(V, h, generator=g, device="cuda") * 0.05).bfloat16()
    y = torch.randint(0, V, (N,), generator=g, device="cuda", dtype=torch.int32)
    G = torch.randn(N, generator=g, device="cuda")
    if N > 1:
        G[torch.rand(N, generator=g, device="cuda") < 0.3] = 0.0
    Hd, Wd, Gd = H.double(), W.double(), G.double()
    z = Hd @ Wd.t()
    l = torch.logsumexp(z, 1)
    dz = -Gd[:, None] * torch.exp(z - l[:, None])
    dz[torch.arange(N, device="cuda"), y.long()] += Gd
    prev = torch.randn(V, h, generator=g, device="cuda")
    want_dH, want_dW = dz @ Wd, dz.t() @ Hd
    ws = sao.workspace(N, h, V)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws)
    cache = sao.logprob_cache(N, V)
    for cached in (False, True):
        dH = torch.full_like(H, float("nan"))
        dW = prev.clone() if accumulate else torch.full((V, h), float("nan"), device="cuda")
        if cached:
            sao.sao_token_logprobs_fwd_cached(H, W, y, logp, lse, cache, ws)
            sao.sao_token_logprobs_bwd_cached(H, W, y, lse, G, dH, dW, cache, ws, accumulate_dW=accumulate)
        else:
            sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws, accumulate_dW=accumulate)
        assert _rel(dH, want_dH) <= TOL
        assert bool((dH[G == 0] == 0).all())
        got = dW.double() - prev.double() if accumulate else dW
        assert _rel(got, want_dW) <= TOL
