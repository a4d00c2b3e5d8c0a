"""fp32 log-probs and their gradient against fp64 (torch on the CPU), at the
edges of the 128x256x32 tiles, with odd hidden sizes, masked rows, several
vocabulary chunks, products cut along their contraction, and operands that the
three-piece splitting cannot represent.

Bounds: a product of two split operands is within 2^-25 of the exact one, sums
of 32 products truncate at most twice at full scale (2^-22), and the K / 32
sums are added in fp32; all relative to sum |a b|, so with u = 2^-24 a
contraction over K terms is off by at most (8 + K / 32) u sum |a b|. On the
random operands here, of random signs, the 2-norm error stays below 16 u, and
1e-5 leaves a factor for exp and the log-sum-exp."""
import numpy as np
import pytest
import torch

from paper_2607_07508_gb300 import sao

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _case(N, h, V, seed=0):
    g = torch.Generator().manual_seed(seed)
    H = torch.randn(N, h, generator=g)
    W = torch.randn(V, h, generator=g) * 0.05
    y = torch.randint(0, V, (N,), generator=g, dtype=torch.int32)
    G = torch.randn(N, generator=g)
    G[torch.rand(N, generator=g) < 0.3] = 0.0
    mask = (torch.rand(N, generator=g) < 0.7).to(torch.uint8)
    return H, W, y, G, mask


def _want(H, W, y, G, lse=None):
    Hd, Wd, Gd = H.double(), W.double(), G.double()
    z = Hd @ Wd.t()
    l = torch.logsumexp(z, 1)
    lp = z.gather(1, y.long()[:, None]).squeeze(1) - l
    dz = -Gd[:, None] * torch.exp(z - l[:, None])
    dz[torch.arange(len(y)), y.long()] += Gd
    act = G != 0
    return lp, l, dz @ Wd, dz[act].t() @ Hd[act]


def _run(H, W, y, G, mask=None, prev=None, offset=0):
    N, h = H.shape
    V = W.shape[0]

    def dev(t):  # `offset` floats past a 256-byte boundary
        flat = torch.empty(t.numel() + offset, dtype=t.dtype, device="cuda")
        out = flat[offset:].view(t.shape)
        out.copy_(t)
        return out
    H, W, y, G = dev(H), dev(W), y.cuda(), G.cuda()
    ws = sao.workspace(N, h, V, torch.float32)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws, row_mask=mask.cuda() if mask is not None else None)
    out = [logp.cpu(), lse.cpu()]
    if mask is None:
        dH = torch.full((N, h), float("nan"), device="cuda")
        dW = prev.clone().cuda() if prev is not None else torch.full((V, h), float("nan"), device="cuda")
        sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws, accumulate_dW=prev is not None)
        out += [dH.cpu(), dW.cpu()]
    return out


def _rel(got, want):
    return float((got.double() - want).norm() / want.norm().clamp(min=1e-300))


@pytest.mark.parametrize("N,h,V,offset", [(1, 1, 2, 0), (127, 31, 129, 0), (128, 32, 128, 0), (129, 33, 127, 1),
                                          (300, 515, 1000, 0), (65, 96, 5000, 1), (1500, 64, 260, 0),
                                          (128, 40, 152 * 256, 0), (129, 40, 77 * 256, 1)])
def test_f32_against_fp64(N, h, V, offset):
    H, W, y, G, mask = _case(N, h, V, seed=N)
    if N == 1:
        G[:] = 0.5
    lp, l, dH, dW = _want(H, W, y, G)
    got = _run(H, W, y, G, offset=offset)
    for g, w in zip(got, (lp, l, dH, dW)):
        assert _rel(g, w) <= TOL
    assert bool((got[2][G == 0] == 0).all())
    glp, gl = _run(H, W, y, G, mask=mask)
    m = mask.bool()
    assert bool((glp[~m] == 0).all()) and bool((gl[~m] == 0).all())
    if m.any():
        assert _rel(glp[m], lp[m]) <= TOL and _rel(gl[m], l[m]) <= TOL


def test_f32_vocabulary_chunks_and_accumulation():
    H, W, y, G, _ = _case(700, 72, 1500, seed=3)
    prev = torch.randn(1500, 72)
    lp, l, dH, dW = _want(H, W, y, G)
    sao.sao_set_dz_budget_bytes(1 << 20)  # below 256 columns of 768 rows: the smallest chunk, 256 columns
    try:
        got = _run(H, W, y, G, prev=prev)
    finally:
        sao.sao_set_dz_budget_bytes(4 << 30)
    assert _rel(got[2], dH) <= TOL and _rel(got[3].double() - prev.double(), dW) <= 2 * TOL


@pytest.mark.parametrize("N", [129, 700])
def test_f32_forward_in_vocabulary_chunks(N):
    """W split 256 rows at a time: six chunks, the last one ragged, with sampled tokens in each."""
    h, V = 520, 1500
    H, W, y, G, mask = _case(N, h, V, seed=4)
    y[:6] = torch.tensor([0, 255, 256, 1279, 1280, 1499], dtype=torch.int32)
    mask[:6] = 1
    prev = torch.randn(V, h)
    lp, l, dH, dW = _want(H, W, y, G)
    assert all(((y >= v) & (y < v + 256)).any() for v in range(0, V, 256))
    sao.sao_set_dz_budget_bytes(1 << 20)  # 6 h bytes a row of W: 256 rows
    try:
        got = _run(H, W, y, G, prev=prev)
        glp, gl = _run(H, W, y, G, mask=mask)
    finally:
        sao.sao_set_dz_budget_bytes(4 << 30)
    assert _rel(got[0], lp) <= TOL and _rel(got[1], l) <= TOL
    assert _rel(got[2], dH) <= TOL and _rel(got[3].double() - prev.double(), dW) <= 2 * TOL
    m = mask.bool()
    assert bool((glp[~m] == 0).all()) and bool((gl[~m] == 0).all())
    assert _rel(glp[m], lp[m]) <= TOL and _rel(gl[m], l[m]) <= TOL


@pytest.mark.parametrize("value", [-3.4028234e38, float("-inf"), float("nan"), 2.0 ** 100])
def test_f32_operands_outside_the_splitting(value):
    """A vocabulary row masked through a bias column, or a NaN: as fp32 gives it."""
    H, W, y, G, _ = _case(200, 40, 300, seed=5)
    H[:, -1] = 1.0
    W[7] = 0.0
    W[7, -1] = value
    if value > 0:
        H[:, -1] = 2.0 ** -100
    y[y == 7] = 8
    lp, l, dH, dW = _want(H, W, y, G)
    got = _run(H, W, y, G)
    assert torch.equal(torch.isnan(got[0]), torch.isnan(lp))
    if not np.isnan(value):
        assert _rel(got[0], lp) <= TOL and _rel(got[1], l) <= TOL
        assert _rel(got[3], dW) <= TOL
    if np.isfinite(value):
        assert _rel(got[2], dH) <= TOL


@pytest.mark.parametrize("N,h,V,offset,budget", [(129, 33, 127, 1, 4 << 30), (300, 516, 1000, 0, 4 << 30),
                                                 (700, 72, 1500, 0, 1 << 20), (1, 4, 257, 0, 4 << 30),
                                                 (130, 17, 20000, 1, 4 << 30)])
def test_f32_fall_back_tiles(N, h, V, offset, budget):
    """The fp32 FMA tiles at the edges of their 128x256x16 shape, with rows on and
    off 16-byte alignment, several vocabulary chunks and products in parts."""
    H, W, y, G, mask = _case(N, h, V, seed=N + h)
    H[:, -1] = 1.0
    W[7] = 0.0
    W[7, -1] = -3.4028234e38
    y[y == 7] = 8
    G[0] = 0.7
    prev = torch.randn(V, h)
    lp, l, dH, dW = _want(H, W, y, G)
    sao.sao_set_dz_budget_bytes(budget)
    try:
        got = _run(H, W, y, G, prev=prev, offset=offset)
        glp, gl = _run(H, W, y, G, mask=mask, offset=offset)
    finally:
        sao.sao_set_dz_budget_bytes(4 << 30)
    assert _rel(got[0], lp) <= TOL and _rel(got[1], l) <= TOL
    assert _rel(got[2], dH) <= TOL and _rel(got[3].double() - prev.double(), dW) <= 2 * TOL
    m = mask.bool()
    assert bool((glp[~m] == 0).all())
    if m.any():
        assert _rel(glp[m], lp[m]) <= TOL and _rel(gl[m], l[m]) <= TOL


def test_f32_fall_back_rate():
    """The fall-back keeps the rate of plain FMA kernels, which did all fp32 heads before: its
    four products in at most three times a matrix library's time for four such products
    (2.3 measured at any clock; FMA kernels of 64x64 tiles 2.7; with operands fetched by the
    computing threads 4.2)."""
    N, h, V = 2048, 1024, 16384
    H, W, y, G, _ = _case(N, h, V, seed=9)
    G[G == 0] = 0.1
    H, W, y, G = H.cuda(), W.cuda(), y.cuda(), G.cuda()
    Z = torch.empty(N, V, device="cuda")
    ws = sao.workspace(N, h, V, torch.float32)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    dH, dW = torch.empty_like(H), torch.empty_like(W)

    def head():
        sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws)
        sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws)

    def least_ms(call):
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert not torch.backends.cuda.matmul.allow_tf32
    product = least_ms(lambda: torch.matmul(H, W.t(), out=Z))
    W[7, 0] = float("-inf")
    assert least_ms(head) <= 3.0 * 4 * product


@pytest.mark.parametrize("e", [25, 61, 63, 70, 90, 99])
def test_f32_products_beyond_fp32(e):
    """H and W each inside the splitting's range, their product beyond fp32's: a
    vocabulary row whose logit is far below the others, or -inf, leaves the rest finite."""
    H, W, y, G, _ = _case(100, 40, 300, seed=e)
    g = torch.Generator().manual_seed(e)
    H[:, 0] = (1 + torch.rand(100, generator=g)) * 2.0 ** e
    W[:, 0] = 0.0
    W[[7, 9]] = 0.0
    W[7, 0], W[9, 0] = -1.37 * 2.0 ** e, -1.61 * 2.0 ** e
    y[(y == 7) | (y == 9)] = 8
    lp, l, dH, dW = _want(H, W, y, G)
    for got, want in zip(_run(H, W, y, G), (lp, l, dH, dW)):
        assert _rel(got, want) <= TOL


@pytest.mark.parametrize("e", [-90, -112])
def test_f32_small_gradients(e):
    """Uniformly small incoming gradients. With dZ above 2^-110 (2^-90 times probabilities of
    1e-3 to 1e-5) its pieces are exact; below, an element is off by 2^-134 at most, so a sum
    over the vocabulary by 2^-134 sum |W|, doubled here for the sums' own rounding to fp32."""
    H, W, y, G, _ = _case(300, 96, 1000, seed=11)
    G *= 2.0 ** e
    lp, l, dH, dW = _want(H, W, y, G)
    got = _run(H, W, y, G)
    for g, want, other in ((got[2], dH, W.double().abs().sum(0)), (got[3], dW, H.double().abs().sum(0))):
        lost = 2.0 ** -133 * other.max() * want.numel() ** 0.5 if e < -100 else 0.0
        assert float((g.double() - want).norm()) <= 1e-6 * float(want.norm()) + lost


def test_f32_gradient_outside_the_splitting():
    """A huge incoming gradient makes dZ leave the splitting's range after the logits stayed inside it."""
    H, W, y, G, _ = _case(150, 40, 300, seed=6)
    G[3] = 1e33
    lp, l, dH, dW = _want(H, W, y, G)
    got = _run(H, W, y, G)
    assert _rel(got[2], dH) <= TOL and _rel(got[3], dW) <= TOL


def test_f32_gradient_outside_the_splitting_with_sms_held():
    """One row's dZ leaves the splitting's range while long one-CTA-per-row
    softmax rows hold 64 SMs, so that some CTAs of the dZ launch start after others
    have raised the flag: every tile is still written, as on an idle GPU."""
    N, h, V = 1024, 32, 8192  # 256 tiles: a CTA on every SM
    H, W, y, G, _ = _case(N, h, V, seed=8)
    G[3] = 1e32
    H, W, y, G = H.cuda(), W.cuda(), y.cuda(), G.cuda()
    ws = sao.workspace(N, h, V, torch.float32)
    logp, lse = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    sao.sao_token_logprobs_fwd(H, W, y, logp, lse, ws)
    long_rows = torch.randn(64, 1 << 22, device="cuda")
    out, side = torch.empty_like(long_rows), torch.cuda.Stream()

    def run(hold):
        dH, dW = torch.empty_like(H), torch.empty_like(W)
        ws[256:].fill_(0xFF)  # a plane that nobody writes reads as NaN
        torch.cuda.synchronize()
        if hold:
            with torch.cuda.stream(side):
                torch.softmax(long_rows, 1, out=out)
        sao.sao_token_logprobs_bwd(H, W, y, lse, G, dH, dW, ws)
        torch.cuda.synchronize()
        return dH, dW

    want = run(False)
    for _ in range(3):
        got = run(True)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
