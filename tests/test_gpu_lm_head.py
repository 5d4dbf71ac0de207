"""GPU parity: row statistics straight from the LM head (tcgen05 GEMM with the
statistics in its epilogue) against the oracle, and against the confidence
kernel run on the materialised logits."""
import numpy as np
import pytest
import torch

from helpers import PROB_ATOL, cuda
from paper_2608_08721_gb300 import binding as lr

pytestmark = pytest.mark.gpu


def _inputs(M, V, Dm, seed, sigma=4.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    H = torch.randn((M, Dm), generator=g, device=cuda()).to(torch.bfloat16)
    W = (torch.randn((V, Dm), generator=g, device=cuda()) * (sigma / Dm ** 0.5)).to(torch.bfloat16)
    return H, W


def _check(orc, H, W, T, rows_per_seq, tok, out):
    row_stat, arg, tp = (None if x is None else x.cpu().numpy() for x in out)
    mx, Z, rarg, rtp, flag = orc.lm_head_stats(H, W, T, rows_per_seq, tok)
    np.testing.assert_allclose(row_stat[:, 0], mx, rtol=1e-5, atol=1e-4)
    np.testing.assert_allclose(row_stat[:, 1], Z, rtol=1e-4)
    bad = (arg != rarg) & (flag == 0)
    assert not bad.any(), np.nonzero(bad)[0]
    if tp is not None:
        np.testing.assert_allclose(tp, rtp, rtol=0, atol=PROB_ATOL)
    return flag


@pytest.mark.parametrize("M,V,Dm", [(33, 32000, 512), (16, 1003, 256), (300, 5000, 128), (128, 4096, 4096),
                                    (17, 128256, 256)])
def test_lm_head_stats_match_oracle(orc, M, V, Dm):
    H, W = _inputs(M, V, Dm, seed=M + V % 97 + Dm)
    rps = 1 if M % 3 else 3
    T = torch.tensor([[0.0, 0.7, 1.0, 1.8][i % 4] for i in range(M // rps)], device=cuda())
    rng = np.random.default_rng(M)
    tok = rng.integers(-1, V, size=M).astype(np.int32)
    ws = lr.LmHeadWorkspace(M, V)
    out = lr.libraspec_lm_head_stats(H, W, ws, temperature=T, rows_per_seq=rps,
                                     tokens=torch.from_numpy(tok).to(cuda()))
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    flag = _check(orc, H, W, T.cpu().numpy(), rps, tok, out)
    assert flag.sum() <= max(1, M // 20)


def test_lm_head_stats_without_tokens_or_temperature(orc):
    H, W = _inputs(40, 3000, 192, seed=4)
    ws = lr.LmHeadWorkspace(40, 3000)
    out = lr.libraspec_lm_head_stats(H, W, ws)
    torch.cuda.synchronize()
    assert out[2] is None
    _check(orc, H, W, None, 1, None, out)


def test_lm_head_confidence_equals_confidence_kernel_on_logits():
    """With the drafter rows and tokens, token_prob / row_stat are the conf /
    dstat that libraspec_confidence computes from the materialised logits."""
    B, K, V, Dm = 4, 16, 32000, 1024
    H, W = _inputs(B * K, V, Dm, seed=9)
    logits = (H.float() @ W.float().T).reshape(B, K, V).contiguous()
    g = torch.Generator(device="cuda").manual_seed(1)
    tok = torch.randint(0, V, (B, K), generator=g, device=cuda(), dtype=torch.int32)
    tok[:, ::2] = logits.argmax(-1)[:, ::2].int()     # high-probability drafts too
    T = torch.tensor([0.0, 1.0, 0.6, 1.4], device=cuda())
    ws = lr.LmHeadWorkspace(B * K, V)
    row_stat, _, tp = lr.libraspec_lm_head_stats(H, W, ws, temperature=T, rows_per_seq=K, tokens=tok.reshape(-1))
    ws2 = lr.Workspace(B, K, V, device=cuda())
    conf, dstat = lr.libraspec_confidence(logits, tok, T, ws2)
    torch.cuda.synchronize()
    np.testing.assert_allclose(tp.reshape(B, K).cpu().numpy(), conf.cpu().numpy(), rtol=0, atol=PROB_ATOL)
    np.testing.assert_allclose(row_stat.reshape(B, K, 2)[..., 0].cpu().numpy(), dstat[..., 0].cpu().numpy(),
                               rtol=1e-5, atol=1e-4)
    np.testing.assert_allclose(row_stat.reshape(B, K, 2)[..., 1].cpu().numpy(), dstat[..., 1].cpu().numpy(),
                               rtol=1e-4)


def test_lm_head_bad_token_sets_status():
    H, W = _inputs(8, 1000, 64, seed=2)
    ws = lr.LmHeadWorkspace(8, 1000)
    tok = torch.zeros(8, dtype=torch.int32, device=cuda())
    tok[3] = 1000
    _, _, tp = lr.libraspec_lm_head_stats(H, W, ws, tokens=tok)
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) & lr.ST_BAD_TOKEN
    assert np.isnan(tp[3].item()) and np.isfinite(tp[:3].cpu().numpy()).all()


def test_lm_head_rejects_unsupported_model_dim():
    H, W = _inputs(4, 100, 64, seed=3)
    ws = lr.LmHeadWorkspace(4, 100)
    with pytest.raises(lr.LibraspecError):
        lr.libraspec_lm_head_stats(H[:, :48].contiguous(), W[:, :48].contiguous(), ws)


def test_lm_head_single_row_and_single_tile_vocabulary(orc):
    for M, V in ((1, 77), (1, 128), (129, 64)):
        H, W = _inputs(M, V, 64, seed=M * 1000 + V)
        ws = lr.LmHeadWorkspace(M, V)
        tok = torch.arange(M, dtype=torch.int32, device=cuda()) % V
        out = lr.libraspec_lm_head_stats(H, W, ws, tokens=tok)
        torch.cuda.synchronize()
        assert lr.libraspec_get_status(ws) == 0
        _check(orc, H, W, None, 1, tok.cpu().numpy(), out)


@pytest.mark.parametrize("M,V,Dm", [(31, 130, 64), (32, 257, 192), (64, 40000, 128), (255, 300, 64), (256, 20011, 64),
                                    (257, 129, 128), (288, 1000, 192), (513, 513, 128), (1100, 700, 64)])
def test_lm_head_tile_edges(orc, M, V, Dm):
    """Row tiles of 32 to 256 rows (one, and several of two sizes), vocabulary ranges with short last tiles and
    columns past the last range, odd and even numbers of k-slabs. Tolerances as in _check: fp32 sums of Dm products."""
    H, W = _inputs(M, V, Dm, seed=M * 31 + V + Dm)
    rng = np.random.default_rng(M + V)
    tok = rng.integers(-1, V, size=M).astype(np.int32)
    tok[:2] = (0, V - 1)
    T = torch.tensor([[0.0, 0.7, 1.3][i % 3] for i in range(M)], device=cuda())
    ws = lr.LmHeadWorkspace(M, V)
    for _ in range(2):  # a workspace is used again as it was left
        out = lr.libraspec_lm_head_stats(H, W, ws, temperature=T, tokens=torch.from_numpy(tok).to(cuda()))
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    flag = _check(orc, H, W, T.cpu().numpy(), 1, tok, out)
    assert flag.sum() <= max(1, M // 20)


@pytest.mark.parametrize("M,V", [(3, 20), (40, 40000), (300, 129 * 128 + 1)])
def test_lm_head_merge_of_steep_and_flat_rows(M, V):
    """Logits that are exact in fp32 (h_m s_v), tile maxima apart by 0 to 4000 in units of log2: Z and the token
    probability against binary64. Tolerance: a term's argument |a| <= 32 (smaller terms are below 2^-32 of Z, at most
    V of them) is rounded by 2^-24 |a| ln 2 = 1.3e-6, ex2.approx adds 2^-22, the sum of 32 terms 9 x 2^-24; those sums
    are added in two floats (2^-39)."""
    g = np.random.default_rng(M + V)
    s = (-g.integers(0, 256, size=V) / 4).astype(np.float32)
    s[: V // 2] -= 64.0  # (whole tiles far below the others)
    s = torch.from_numpy(s).to(torch.bfloat16)
    h = torch.tensor([[0.0, 0.25, 1.0, 2.0, 16.0][i % 5] for i in range(M)])
    T = torch.tensor([[1.0, 0.7, 0.0][i % 3] for i in range(M)])
    tok = g.integers(0, V, size=M).astype(np.int32)
    H, W = torch.zeros(M, 64), torch.zeros(V, 64)
    H[:, 5], W[:, 5] = h, s.float()
    ws = lr.LmHeadWorkspace(M, V)
    stat, arg, tp = lr.libraspec_lm_head_stats(H.to(cuda(), torch.bfloat16), W.to(cuda(), torch.bfloat16), ws,
                                               temperature=T.to(cuda()), tokens=torch.from_numpy(tok).to(cuda()))
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    x = np.outer(h.numpy().astype(np.float64), s.float().numpy().astype(np.float64))
    c = np.where(T.numpy() > 0, 1 / np.maximum(T.numpy().astype(np.float64), 1e-9), 1.0)[:, None]
    mx = x.max(1)
    e = np.exp((x - mx[:, None]) * c)
    Z = e.sum(1)
    assert (arg.cpu().numpy() == x.argmax(1)).all()
    assert (stat[:, 0].cpu().numpy() == mx).all()
    np.testing.assert_allclose(stat[:, 1].cpu().numpy(), Z, rtol=2.5e-6)
    p = e[np.arange(M), tok] / Z
    np.testing.assert_allclose(tp.cpu().numpy(), p, rtol=3e-6, atol=1.5e-45)


@pytest.mark.parametrize("M", [1, 33, 200, 300])
def test_lm_head_sum_keeps_small_terms_beside_a_large_one(M):
    """One column of each row weighs 1 and every other 2^-32 (T = log2(e): logits in units of log2): every power and
    every product is exact, so Z has its last rounding alone, 2^-24. A CTA's 128 columns add 2^-25 to the 1, which a
    sum in 32 bits over its six or seven tiles would drop each time."""
    V = 128256
    s = torch.full((V, M), -32.0)
    at = torch.arange(M) * 379 % V  # (in every tile of a CTA's columns)
    s[at, torch.arange(M)] = 0.0
    D = (M + 63) // 64 * 64
    H, W = torch.eye(M, D), torch.zeros(V, D)
    W[:, :M] = s
    T = torch.full((M,), float(np.float32(np.log2(np.e))))
    ws = lr.LmHeadWorkspace(M, V)
    stat, arg, tp = lr.libraspec_lm_head_stats(H.to(cuda(), torch.bfloat16), W.to(cuda(), torch.bfloat16), ws,
                                               temperature=T.to(cuda()), tokens=at.int().to(cuda()))
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    Z = 1.0 + (V - 1) * 2.0 ** -32
    assert (arg.cpu() == at).all() and (stat[:, 0] == 0).all()
    assert np.abs(stat[:, 1].cpu().numpy().astype(np.float64) / Z - 1).max() <= 2.0 ** -24
    assert np.abs(tp.cpu().numpy().astype(np.float64) * Z - 1).max() <= 2.0 ** -24
