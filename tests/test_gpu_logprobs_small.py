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


@pytest.mark.parametrize("N,offset", [(15, 0), (17, 0), (4095, 0), (4096, 1), (4097, 0), (8192, 0), (8193, 0),
                                      (12305, 1)])
def test_row_lists_and_merge(N, offset):
    """Rows listed by mask and by gradient at the edges of the 16-row threads and
    4,096-row blocks, with arrays one element off alignment, and the merge of the
    tile partials with a warp and with eight threads per row."""
    h, V = 8, 700
    g = torch.Generator(device="cuda").manual_seed(N)

    def shifted(t):
        out = torch.empty(t.numel() + offset, dtype=t.dtype, device="cuda")[offset:]
        return out.copy_(t)
    H = torch.randn(N, h, generator=g, device="cuda").bfloat16()
    W = (torch.randn(V, h, generator=g, device="cuda") * 0.3).bfloat16()
    y = torch.randint(0, V, (N,), generator=g, device="cuda", dtype=torch.int32)
    mask = shifted((torch.rand(N, generator=g, device="cuda") < 0.6).to(torch.uint8))
    G = shifted(torch.randn(N, generator=g, device="cuda") * (torch.rand(N, generator=g, device="cuda") < 0.5))
    Hd, Wd = H.double(), W.double()
    z = Hd @ Wd.t()
    l = torch.logsumexp(z, 1)
    lp = z.gather(1, y.long()[:, None]).squeeze(1) - l
    dz = -G.double()[:, None] * torch.exp(z - l[:, None])
    dz[torch.arange(N, device="cuda"), y.long()] += G.double()
    ws = sao.workspace(N, h, V)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws, row_mask=mask)
    m = mask.bool()
    assert float((logp[m].double() - lp[m]).abs().max()) <= 1e-4 and bool((logp[~m] == 0).all())
    sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws)
    assert float((lse.double() - l).abs().max()) <= 1e-4
    dH, dW = torch.empty_like(H), torch.empty(V, h, device="cuda")
    sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws)
    assert _rel(dH, dz @ Wd) <= TOL and _rel(dW, dz.t() @ Hd) <= TOL
    assert bool((dH[G == 0] == 0).all())


@pytest.mark.parametrize("V", [256, 257, 543, 1024])
def test_epilogue_column_paths(V):
    """Sampled tokens at the edges of the 32-column chunks, vocabularies that end
    inside a chunk and at its edge, rows without gradient, sampled tokens far
    below their row's maximum (flagged in the cached forward), and a NaN row of H
    without gradient, which must not reach the others."""
    N, h = 130, 72
    g = torch.Generator(device="cuda").manual_seed(V)
    H = torch.randn(N, h, generator=g, device="cuda").bfloat16()
    W = (torch.randn(V, h, generator=g, device="cuda") * 0.3).bfloat16()
    y = torch.tensor([[0, 1, 31, 32, 63, 64, 255, V - 2, V - 1][i % 9] for i in range(N)], dtype=torch.int32,
                     device="cuda")
    H[5] = W[40] * (90.0 / float(W[40].double() @ W[40].double()))  # z[5, 40] = 90, the sampled token's near 0
    G = torch.randn(N, generator=g, device="cuda")
    G[::7] = 0.0
    mask = torch.ones(N, dtype=torch.uint8, device="cuda")
    mask[7] = 0
    H[7] = float("nan")
    ok = mask.bool()
    Hd, Wd, Gd = torch.where(ok[:, None], H.double(), 0.0), W.double(), G.double()
    z = Hd @ Wd.t()
    l = torch.logsumexp(z, 1)
    lp = z.gather(1, y.long()[:, None]).squeeze(1) - l
    dz = -Gd[:, None] * torch.exp(z - l[:, None])
    dz[torch.arange(N, device="cuda"), y.long()] += Gd
    ws = sao.workspace(N, h, V)
    for cached in (False, True):
        logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
        dH, dW = torch.empty_like(H), torch.empty(V, h, device="cuda")
        if cached:
            cache = sao.logprob_cache(N, V)
            sao.sao_token_logprobs_fwd_cached(H, W, y, logp, lse, cache, ws, row_mask=mask)
            sao.sao_token_logprobs_bwd_cached(H, W, y, lse, G, dH, dW, cache, ws)
        else:
            sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws, row_mask=mask)
            sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws)
        # fp32 sums of h products and V exponentials of logits up to 90
        assert float((logp[ok].double() - lp[ok]).abs().max()) <= 2e-4
        assert _rel(dH, dz @ Wd) <= TOL and _rel(dW, dz.t() @ Hd) <= TOL


@pytest.mark.parametrize("V", [4096 + 40, 4096 + 64, 2 * 4096 + 200, 4096])
def test_parts_of_a_short_last_chunk(V):
    """The dZ buffer holds 4,096 vocabulary columns at a time and dH's product is
    cut into parts: a last chunk with fewer 64-column blocks than parts leaves
    some parts empty, and they add nothing."""
    N, h = 128, 72
    g = torch.Generator(device="cuda").manual_seed(V)
    H = torch.randn(N, h, generator=g, device="cuda").bfloat16()
    W = (torch.randn(V, h, generator=g, device="cuda") * 0.3).bfloat16()
    y = torch.randint(0, V, (N,), generator=g, device="cuda", dtype=torch.int32)
    G = torch.randn(N, generator=g, device="cuda")
    Hd, Wd, Gd = H.double(), W.double(), G.double()
    z = Hd @ Wd.t()
    dz = -Gd[:, None] * torch.exp(z - torch.logsumexp(z, 1)[:, None])
    dz[torch.arange(N, device="cuda"), y.long()] += Gd
    before = sao.sao_get_dz_budget_bytes()
    sao.sao_set_dz_budget_bytes(N * 4096 * 2)
    try:
        ws = sao.workspace(N, h, V)
        logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
        dH, dW = torch.full_like(H, float("nan")), torch.full((V, h), float("nan"), device="cuda")
        sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws)
        sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws)
        assert _rel(dH, dz @ Wd) <= TOL and _rel(dW, dz.t() @ Hd) <= TOL
    finally:
        sao.sao_set_dz_budget_bytes(before)


def test_cached_rows_are_scaled_after_their_parts_are_added():
    """dH of stored rows is a scale times a sum cut into parts: an infinite incoming
    gradient gives infinities of the sum's signs, not the sum of infinities."""
    N, h, V = 11, 64, 4000  # one tile of K = 4,000: seven parts
    g = torch.Generator(device="cuda").manual_seed(1)
    H = torch.randn(N, h, generator=g, device="cuda").bfloat16()
    W = (torch.randn(V, h, generator=g, device="cuda") * 0.3).bfloat16()
    y = torch.randint(0, V, (N,), generator=g, device="cuda", dtype=torch.int32)
    ws, cache = sao.workspace(N, h, V), sao.logprob_cache(N, V)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    sao.sao_token_logprobs_fwd_cached(H, W, y, logp, lse, cache, ws)
    dW, got = torch.empty(V, h, device="cuda"), []
    for top in (1.0, float("inf")):
        G = torch.ones(N, device="cuda")
        G[3] = top
        dH = torch.empty_like(H)
        sao.sao_token_logprobs_bwd_cached(H, W, y, lse, G, dH, dW, cache, ws)
        got.append(dH.float())
    assert bool((got[0][3] != 0).all()) and torch.equal(got[1][3], got[0][3] * float("inf"))
    rest = torch.arange(N, device="cuda") != 3
    assert torch.equal(got[0][rest], got[1][rest])
