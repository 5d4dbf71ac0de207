"""GPU parity: block-causal GQA verify attention vs. the fp64 oracle."""
import numpy as np
import pytest
import torch

from helpers import check_attn, cuda
from paper_2608_08721_gb300 import binding as lr
from paper_2608_08721_gb300 import workloads

pytestmark = pytest.mark.gpu


def _inputs(B, K, Hq, Hkv, d, kv, S_cap, seed, scale_k=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    Q = torch.randn((B, K + 1, Hq, d), generator=g, device=cuda()).to(torch.bfloat16)
    Kc = (torch.randn((B, Hkv, S_cap, d), generator=g, device=cuda()) * scale_k).to(torch.bfloat16)
    Vc = torch.randn((B, Hkv, S_cap, d), generator=g, device=cuda()).to(torch.bfloat16)
    return Q, Kc, Vc


def _run(Q, Kc, Vc, kv, L, K):
    B, _, Hq, d = Q.shape
    Hkv, S_cap = Kc.shape[1], Kc.shape[2]
    ws = lr.Workspace(B, K, 1, Hq, Hkv, d, S_cap, device=cuda())
    kv_t = torch.tensor(kv, dtype=torch.int32, device=cuda())
    L_t = torch.tensor(L, dtype=torch.int32, device=cuda())
    O, lse = lr.libraspec_verify_attn(Q, Kc, Vc, kv_t, L_t, ws, want_lse=True)
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    return O, lse


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,Hkv", [(8, 2), (28, 4), (32, 8), (64, 8), (4, 4)])
def test_attn_small_ragged(orc, d, Hq, Hkv):
    K = 9
    kv = [0, 1, 63, 64, 200, 700]
    L = [0, 9, 3, 1, 9, 5]
    B = len(kv)
    S_cap = max(k + l + 1 for k, l in zip(kv, L)) + 3
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, kv, S_cap, seed=Hq * 7 + d, scale_k=2.0)
    O, lse = _run(Q, Kc, Vc, kv, L, K)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array(kv), np.array(L))
    check_attn(O, lse, O_ref, lse_ref, L)


def test_attn_rows_beyond_L_untouched():
    K, B, Hq, Hkv, d = 6, 2, 8, 2, 64
    kv, L = [30, 5], [2, 0]
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, kv, 48, seed=1)
    ws = lr.Workspace(B, K, 1, Hq, Hkv, d, 48, device=cuda())
    O = torch.full_like(Q, 7.0)
    lr.libraspec_verify_attn(Q, Kc, Vc, torch.tensor(kv, dtype=torch.int32, device=cuda()),
                             torch.tensor(L, dtype=torch.int32, device=cuda()), ws, O=O)
    torch.cuda.synchronize()
    assert torch.all(O[0, 3:] == 7.0) and torch.all(O[1, 1:] == 7.0)
    assert not torch.any(O[0, :3] == 7.0)


@pytest.mark.parametrize("kv", [5000, 20000])
def test_attn_long_split_kv_merge(orc, kv):
    # one sequence, long cache: its row groups spread over many CTAs and are merged
    K, Hq, Hkv, d = 16, 32, 8, 128
    L = [11]
    Q, Kc, Vc = _inputs(1, K, Hq, Hkv, d, [kv], kv + K + 1, seed=kv)
    O, lse = _run(Q, Kc, Vc, [kv], L, K)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array([kv]), np.array(L))
    check_attn(O, lse, O_ref, lse_ref, L)


@pytest.mark.parametrize("kv", [300, 20000])
@pytest.mark.parametrize("Hq,Hkv,d,L", [(32, 8, 128, 7), (32, 8, 64, 3), (64, 8, 128, 3), (8, 8, 128, 16),
                                        (32, 8, 128, 12)])
def test_attn_small_groups_long_cache(orc, kv, Hq, Hkv, d, L):
    """Row groups of 16 to 52 rows (a few block positions of g heads) over a
    short and a long cache: one CTA per group, and groups split over many
    CTAs whose parts are merged."""
    K = 16
    Q, Kc, Vc = _inputs(1, K, Hq, Hkv, d, [kv], kv + K + 1, seed=kv + Hq + L, scale_k=2.0)
    O, lse = _run(Q, Kc, Vc, [kv], [L], K)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array([kv]), np.array([L]))
    check_attn(O, lse, O_ref, lse_ref, [L])


@pytest.mark.parametrize("d", [64, 128])
def test_attn_small_groups_ragged(orc, d):
    """Several sequences with small row groups of different sizes, some
    covered by one CTA, some split."""
    K, Hq, Hkv = 9, 32, 8
    kv = [0, 3000, 64, 700, 9000]
    L = [7, 0, 3, 5, 1]
    S_cap = max(k + l + 1 for k, l in zip(kv, L)) + 3
    Q, Kc, Vc = _inputs(len(kv), K, Hq, Hkv, d, kv, S_cap, seed=d + 5, scale_k=2.0)
    O, lse = _run(Q, Kc, Vc, kv, L, K)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array(kv), np.array(L))
    check_attn(O, lse, O_ref, lse_ref, L)


def test_attn_peaky_scores(orc):
    w = workloads.WORKLOADS["sampling"].scaled(B=4, kv=("uniform", 100, 3000))
    kv = workloads.kv_lengths(w)
    lay = workloads.layer(w, 0, kv, device=cuda(), peaky=True)
    L = np.array([0, 16, 7, 3], np.int32)
    O, lse = _run(lay["Q"], lay["Kc"], lay["Vc"], kv.tolist(), L.tolist(), w.K)
    O_ref, lse_ref = orc.verify_attn(lay["Q"], lay["Kc"], lay["Vc"], kv, L)
    check_attn(O, lse, O_ref, lse_ref, L)


def test_attn_equal_keys_closed_form():
    # all keys equal: every row's output is the mean of its visible values
    B, K, Hq, Hkv, d = 1, 4, 4, 1, 64
    kv = [100]
    L = [4]
    S = 128
    g = torch.Generator(device="cuda").manual_seed(3)
    Q = torch.randn((B, K + 1, Hq, d), generator=g, device=cuda()).to(torch.bfloat16)
    Kc = torch.full((B, Hkv, S, d), 0.25, device=cuda(), dtype=torch.bfloat16)
    Vc = torch.randn((B, Hkv, S, d), generator=g, device=cuda()).to(torch.bfloat16)
    O, _ = _run(Q, Kc, Vc, kv, L, K)
    for t in range(5):
        mean = Vc[0, 0, : kv[0] + t + 1].float().mean(0)
        for h in range(Hq):
            assert torch.allclose(O[0, t, h].float(), mean, atol=1e-2, rtol=1e-2)


@pytest.mark.parametrize("name", ["tiny", "8b", "sampling", "ragged", "70b"])
def test_attn_full_size_sampled_rows(orc, name):
    """One layer at the workload's full size, in the launch configuration the
    benchmark uses; the oracle checks a sample of rows one by one."""
    w = workloads.WORKLOADS[name]
    kv = workloads.kv_lengths(w)
    rng = np.random.default_rng(len(name))
    L = rng.integers(0, w.K + 1, size=w.B).astype(np.int32)
    L[0] = w.K
    if w.B > 1:
        L[1] = 0
    lay = workloads.layer(w, 3, kv, device=cuda())
    O, lse = _run(lay["Q"], lay["Kc"], lay["Vc"], kv.tolist(), L.tolist(), w.K)
    rows = []
    for b in range(w.B):
        for h in rng.choice(w.Hq, size=min(3, w.Hq), replace=False):
            rows.append((b, int(h), int(L[b])))
            rows.append((b, int(h), int(rng.integers(0, L[b] + 1))))
    # complete (sequence, kv head) row groups: every head of the kv head at every verified
    # position, the rows the kernel's split-KV merge writes together (sequence 0 at L = K,
    # so (K + 1) g rows: one full 128-row tile or more; and the last sequence)
    g = w.Hq // w.Hkv
    for b in sorted({0, w.B - 1}):
        kvh = int(rng.integers(0, w.Hkv))
        rows += [(b, kvh * g + i, t) for i in range(g) for t in range(int(L[b]) + 1)]
    rows = np.array(sorted(set(rows)), np.int32)
    O_ref, lse_ref = orc.verify_attn(lay["Q"], lay["Kc"], lay["Vc"], kv, L, rows=rows)
    check_attn(O, lse, O_ref, lse_ref, L, rows=[tuple(r) for r in rows])


def test_attn_kv_overflow_sets_status_and_skips():
    B, K, Hq, Hkv, d, S = 2, 4, 4, 2, 64, 32
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, None, S, seed=2)
    ws = lr.Workspace(B, K, 1, Hq, Hkv, d, S, device=cuda())
    O = torch.zeros_like(Q)
    lr.libraspec_verify_attn(Q, Kc, Vc, torch.tensor([30, 5], dtype=torch.int32, device=cuda()),
                             torch.tensor([4, 4], dtype=torch.int32, device=cuda()), ws, O=O)
    assert lr.libraspec_get_status(ws) & lr.ST_KV_OVERFLOW
    assert torch.all(O[0] == 0) and torch.any(O[1] != 0)


def test_attn_deterministic():
    B, K, Hq, Hkv, d = 3, 16, 32, 8, 128
    kv = [9000, 300, 4000]
    L = [16, 2, 9]
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, kv, 9100, seed=11)
    outs = [_run(Q, Kc, Vc, kv, L, K) for _ in range(3)]
    for b in range(B):
        rows = slice(0, L[b] + 1)   # rows beyond L_b are never written
        for O, lse in outs[1:]:
            assert torch.equal(O[b, rows], outs[0][0][b, rows])
            assert torch.equal(lse[b, rows], outs[0][1][b, rows])


@pytest.mark.parametrize("B,kv_hi,d,seed", [(300, 200, 64, 1), (40, 9000, 128, 2), (129, 64, 128, 3),
                                             (1500, 40, 128, 4)])
def test_attn_many_sequences_stream_k_ranges(orc, B, kv_hi, d, seed):
    """Many ragged sequences: CTA tile ranges start and end inside row groups,
    one CTA covers several whole groups, and groups spread over many CTAs.
    B = 1500 is past the 1024 sequences whose lengths the kernel keeps in
    shared memory for its plan: that batch plans from global memory."""
    rng = np.random.default_rng(seed)
    K, Hq, Hkv = 12, 16, 4
    kv = rng.integers(0, kv_hi + 1, size=B).astype(np.int32)
    L = rng.integers(0, K + 1, size=B).astype(np.int32)
    S_cap = int((kv + L).max()) + 1
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, kv, S_cap, seed=seed * 101)
    rows = np.array([(b, h, t) for b in range(B) for h in (0, Hq - 1) for t in {0, int(L[b])}], np.int32)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, kv, L, rows=rows)
    for _ in range(4):  # repeated: warps of one item race on shared memory if unsynchronised
        O, lse = _run(Q, Kc, Vc, kv.tolist(), L.tolist(), K)
        check_attn(O, lse, O_ref, lse_ref, L, rows=[tuple(r) for r in rows])


@pytest.mark.parametrize("name,n_layers,L_max", [("8b", 4, None), ("sampling", 3, None), ("tiny", 3, None),
                                                 ("8b", 3, 4)])
def test_attn_layer_chain_matches_per_layer_oracle(orc, name, n_layers, L_max):
    """libraspec_verify_attn_layers: all layers in one persistent launch; each
    layer's split groups are merged after the grid barrier that ends it."""
    w = workloads.WORKLOADS[name]
    kv = workloads.kv_lengths(w)
    rng = np.random.default_rng(7)
    L = rng.integers(0, (L_max if L_max is not None else w.K) + 1, size=w.B).astype(np.int32)
    layers = [workloads.layer(w, l, kv, device=cuda()) for l in range(n_layers)]
    S = layers[0]["Kc"].shape[2]
    ws = lr.Workspace(w.B, w.K, 1, w.Hq, w.Hkv, w.d, S, device=cuda())
    outs, lses = lr.libraspec_verify_attn_layers(layers, torch.tensor(kv, device=cuda()),
                                                 torch.tensor(L, device=cuda()), ws, want_lse=True)
    torch.cuda.synchronize()
    assert lr.libraspec_get_status(ws) == 0
    rows = np.array([(b, h, t) for b in range(w.B) for h in (0, w.Hq - 1) for t in {0, int(L[b])}], np.int32)
    for l in range(n_layers):
        O_ref, lse_ref = orc.verify_attn(layers[l]["Q"], layers[l]["Kc"], layers[l]["Vc"], kv, L, rows=rows)
        check_attn(outs[l], lses[l], O_ref, lse_ref, L, rows=[tuple(r) for r in rows])
    # the chain equals one layer at a time
    for l in range(n_layers):
        O1, lse1 = _run(layers[l]["Q"], layers[l]["Kc"], layers[l]["Vc"], kv.tolist(), L.tolist(), w.K)
        for b in range(w.B):
            assert torch.equal(O1[b, : L[b] + 1], outs[l][b, : L[b] + 1])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,Hkv,K", [(16, 2, 16), (32, 8, 32), (14, 2, 17), (8, 8, 8)])
def test_attn_step_and_unit_edges(orc, d, Hq, Hkv, K):
    """Items of one to several 128-key steps whose last is half or full (one stream idle, both, an odd count), and
    row groups of fewer than 128 rows, of exactly 128, and a second group behind them. Tolerances as in check_attn."""
    kv = [0, 62, 63, 64, 127, 128, 129, 191, 255, 256, 257, 320, 500, 1100]
    L = [K, 0, K, K - 1, K - 2, K, 1, K, K // 2, K, 0, K - 1, K, K]
    S_cap = max(kv) + K + 1
    Q, Kc, Vc = _inputs(len(kv), K, Hq, Hkv, d, kv, S_cap, seed=d + Hq + K, scale_k=2.0)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array(kv), np.array(L))
    for _ in range(3):
        O, lse = _run(Q, Kc, Vc, kv, L, K)
        check_attn(O, lse, O_ref, lse_ref, L)


@pytest.mark.parametrize("B,kv,L,Hq,Hkv,d", [(1, 4096, 5, 8, 8, 128), (1, 100, 0, 32, 8, 128), (3, 640, 9, 16, 4, 64),
                                             (5, 63, 3, 8, 2, 128), (40, 200, 12, 16, 4, 64), (2, 9000, 12, 64, 64, 128)])
def test_attn_equal_groups_get_whole_ctas(orc, B, kv, L, Hq, Hkv, d):
    """Equal caches and lengths: each row group has its own CTAs (one that covers it, or several whose parts are
    merged), or, with groups a few too many for that, the batch is cut by cost. Tolerances as in check_attn."""
    K = 16
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, None, kv + K + 1, seed=B * 100 + kv, scale_k=2.0)
    kvs, Ls = [kv] * B, [L] * B
    rows = np.array([(b, h, t) for b in range(B) for h in (0, Hq // 2, Hq - 1) for t in {0, L}], np.int32)
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array(kvs), np.array(Ls), rows=rows)
    for _ in range(2):
        O, lse = _run(Q, Kc, Vc, kvs, Ls, K)
        check_attn(O, lse, O_ref, lse_ref, Ls, rows=[tuple(r) for r in rows])


@pytest.mark.parametrize("n_layers", [1, 2])
@pytest.mark.parametrize("L,Hq,Hkv,kv", [(0, 2, 2, 1900), (1, 8, 2, 1101)])
def test_attn_more_parts_than_rows_on_one_workspace(orc, n_layers, L, Hq, Hkv, kv):
    """Row groups of 1 and 8 rows spread over 30 and 18 CTAs, most of which have no row to merge: the groups' counters
    are left at zero for the next call all the same (new inputs every call). Tolerances as in check_attn."""
    K, d = 4, 64
    S_cap = kv + K + 1
    ws = lr.Workspace(1, K, 1, Hq, Hkv, d, S_cap, device=cuda())
    kv_t = torch.tensor([kv], dtype=torch.int32, device=cuda())
    L_t = torch.tensor([L], dtype=torch.int32, device=cuda())
    for call in range(6):
        layers = [dict(zip(("Q", "Kc", "Vc"), _inputs(1, K, Hq, Hkv, d, None, S_cap, seed=10 * call + l, scale_k=2.0)))
                  for l in range(n_layers)]
        Os, lses = lr.libraspec_verify_attn_layers(layers, kv_t, L_t, ws, want_lse=True)
        torch.cuda.synchronize()
        assert lr.libraspec_get_status(ws) == 0
        for lay, O, lse in zip(layers, Os, lses):
            O_ref, lse_ref = orc.verify_attn(lay["Q"], lay["Kc"], lay["Vc"], np.array([kv]), np.array([L]))
            check_attn(O, lse, O_ref, lse_ref, [L])


@pytest.mark.parametrize("d", [64, 128])
def test_attn_late_rise_of_the_reference_max(orc, d):
    """One key raises a row's max by 2^9 to 2^12 above that of the item's first 32 keys: in each 32-key chunk of a
    128-key step, in the first step of either stream and in later ones, in some rows of a warp and not in others. The
    earlier keys keep a good part of the weight (2^6 each, or large values), so that P, l and O rescaled wrongly show.
    Each of the 128 row groups is one item. Tolerances as in check_attn."""
    K, Hq, Hkv, kv = 16, 16, 4, 520
    at = [33, 47, 63, 64, 65, 95, 96, 100, 127, 160, 163, 191, 192, 222, 224, 255,
          256, 257, 288, 300, 320, 352, 383, 384, 416, 450, 480, 511, 512, 513, 517, 519]
    B, S_cap = len(at), kv + K + 1
    L = [[0, 3, 7, 16][b % 4] for b in range(B)]
    Q, Kc, Vc = _inputs(B, K, Hq, Hkv, d, None, S_cap, seed=d, scale_k=0.1)
    key = torch.arange(S_cap, device=cuda())
    level = torch.where((key < 256) & (key % 128 < 32), 0.0, 6.0).repeat(B, 1)  # in log2 of the weight
    for b, k in enumerate(at):
        level[b, k] = 9.0 + b % 4
    Kc[..., 0] = (level * (d ** 0.5 * np.log(2.0))).to(torch.bfloat16)[:, None, :]
    Q[..., 0] = torch.tensor([1.0, -1.0, 0.9375, 1.0], device=cuda()).repeat(Hq // 4)
    Vc[:, :, :32] += 4.0
    O_ref, lse_ref = orc.verify_attn(Q, Kc, Vc, np.array([kv] * B), np.array(L))
    for _ in range(3):
        O, lse = _run(Q, Kc, Vc, [kv] * B, L, K)
        check_attn(O, lse, O_ref, lse_ref, L)
