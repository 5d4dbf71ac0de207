"""Performance cases of the verify round: the calls a serving loop makes on this library.

Every case goes through the public binding (``paper_2608_08721_gb300.binding``) on device-resident
inputs. Shapes are the repository's own workloads (vocabularies 32000 / 128256 / 152064, GQA 8/2, 32/8,
28/4, 64/8, head dim 64 / 128, batch 1 to 64, caches of 512 to 131072 keys, blocks of 16 / 32 drafted
tokens, draft trees of 16 to 512 nodes); ``draw`` spreads over the ranges between and around them.

Cache lengths and verified lengths come from the case itself (``lens`` seeds them), so that the work of
a case is known from the case; every tensor's values come from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2608_08721_gb300 import binding as lr
from paper_2608_08721_gb300 import workloads

LOG2E = 1.4426950408889634


def listed():
    return [
        # the smallest whole round: one greedy sequence, one layer (GQA 8/2, d 64), where latency and launches count
        dict(name="round_small", kind="round", B=1, K=16, V=32000, Hq=8, Hkv=2, d=64, layers=1, kv_lo=512, kv_hi=512,
             T=0.0, noise=1.0, bf16=False, lens=1),
        # a whole round of a sampling batch (T = 1) on an engine's bf16 logits
        dict(name="round_sampling", kind="round", B=16, K=16, V=152064, Hq=28, Hkv=4, d=128, layers=1, kv_lo=1024,
             kv_hi=8192, T=1.0, noise=1.5, bf16=True, lens=2),
        # drafter confidence and length selection of a full serving batch: one pass over 1 GB of logits
        dict(name="select_batch", kind="select", B=64, K=32, V=128256, T=0.8, noise=1.0, bf16=False, lens=3),
        # decode at batch 1: the 32 attention layers of an 8B-class target over a 4K cache, short draft
        dict(name="attn_b1_layers", kind="attn", B=1, K=16, Hq=32, Hkv=8, d=128, layers=32, kv_lo=4096, kv_hi=4096,
             L_lo=4, L_hi=4, tree=False, page=0, lse=False, lens=4),
        # a mid-size batch on a serving engine's paged cache, log-sum-exp wanted, g = 7
        dict(name="attn_paged", kind="attn", B=16, K=16, Hq=28, Hkv=4, d=128, layers=2, kv_lo=1024, kv_hi=8192,
             L_lo=0, L_hi=16, tree=False, page=128, lse=True, lens=5),
        # a full serving batch with log-uniform cache lengths and short selected lengths
        dict(name="attn_ragged", kind="attn", B=64, K=32, Hq=32, Hkv=8, d=128, layers=1, kv_lo=512, kv_hi=32768,
             L_lo=0, L_hi=7, tree=False, page=0, lse=False, lens=6),
        # long-context decode: 8 sequences over 128K keys, one 70B-class layer (64/8)
        dict(name="attn_long", kind="attn", B=8, K=16, Hq=64, Hkv=8, d=128, layers=1, kv_lo=131072, kv_hi=131072,
             L_lo=1, L_hi=8, tree=False, page=0, lse=False, lens=7),
        # verification of a large draft tree (the largest node budget) over four layers
        dict(name="attn_tree", kind="attn", B=1, K=512, Hq=32, Hkv=8, d=128, layers=4, kv_lo=4096, kv_hi=4096,
             L_lo=512, L_hi=512, tree=True, page=0, lse=False, lens=8),
        # acceptance of a full batch, greedy and sampling sequences mixed
        dict(name="accept_batch", kind="accept", B=64, K=32, V=128256, L_lo=0, L_hi=8, T=0.8, mixed=True, noise=1.0,
             bf16=False, lens=9),
        # the sampling walk of draft trees on bf16 logits
        dict(name="accept_tree", kind="accept_tree", B=2, K=256, V=152064, T=1.0, bf16=True, lens=10),
        # row statistics from the LM head at batch 1: 16 drafter and 17 target rows, the head's bytes bound it
        dict(name="lm_head_decode", kind="lm_head", M=33, V=128256, Dm=4096, rows_per_seq=33, T=0.0),
        # row statistics from the LM head for a full batch: 64 x 33 rows, bound by the tensor cores
        dict(name="lm_head_batch", kind="lm_head", M=2112, V=128256, Dm=4096, rows_per_seq=33, T=0.8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng):
    """A vocabulary of 32000 to 152064: mostly a multiple of 64, as padded heads have, now and then any number."""
    v = _log_int(rng, 32000, 152064)
    return v if rng.random() < 0.25 else min(152064, (v + 63) // 64 * 64)


def _heads(rng):
    return rng.choice([(8, 2), (16, 4), (32, 8), (28, 4), (64, 8), (8, 8), (16, 2), (32, 4)])


def draw(rng):
    kind = rng.choice(["round", "select", "attn", "attn", "attn_tree", "accept", "accept_tree", "lm_head"])
    lens = rng.randrange(1 << 30)
    bf16 = rng.random() < 0.5
    T = rng.choice([0.0, 0.7, 0.8, 1.0])
    noise = round(rng.uniform(0.5, 3.0), 2)
    K = rng.choice([8, 11, 15, 16, 16, 24, 32])
    if kind == "lm_head":
        return dict(kind=kind, M=_log_int(rng, 1, 2112), V=_vocab(rng), Dm=64 * rng.randint(32, 64),
                    rows_per_seq=rng.choice([1, 16, 33]), T=T)
    if kind in ("select", "accept"):
        B = _log_int(rng, 1, 64)
        if kind == "select":
            return dict(kind=kind, B=B, K=K, V=min(_vocab(rng), 128256), T=T, noise=noise, bf16=bf16, lens=lens)
        L_hi = rng.randint(2, min(K, 8))
        return dict(kind=kind, B=B, K=K, V=min(_vocab(rng), 128256), L_lo=0, L_hi=L_hi, T=T or 0.8,
                    mixed=rng.random() < 0.5, noise=noise, bf16=bf16, lens=lens)
    if kind == "accept_tree":
        N = _log_int(rng, 16, 512)
        return dict(kind=kind, B=rng.randint(1, max(1, 512 // N)), K=N, V=_vocab(rng), T=T, bf16=bf16, lens=lens)
    Hq, Hkv = _heads(rng)
    d = rng.choice([64, 128, 128])
    if kind == "attn_tree":
        N = _log_int(rng, 16, 512)
        kv_hi = _log_int(rng, 512, 4096)
        return dict(kind="attn", B=1 if N > 128 else rng.randint(1, 4), K=N, Hq=Hq if Hq <= 32 else 32, Hkv=Hkv, d=d,
                    layers=rng.randint(1, 4), kv_lo=kv_hi // 2, kv_hi=kv_hi, L_lo=max(1, N - 3), L_hi=N, tree=True,
                    page=rng.choice([0, 0, 64, 128]), lse=rng.random() < 0.3, lens=lens)
    B = _log_int(rng, 1, 64)
    kv_hi = _log_int(rng, 512, max(513, min(131072, 1 << 20 if B == 1 else 520000 // B)))
    kv_lo = rng.choice([kv_hi, max(1, kv_hi // 4), max(1, kv_hi // 32)])
    layers = rng.choice([1, 2, 4, 32]) if B * kv_hi <= 16384 else rng.choice([1, 2])
    if kind == "round":
        return dict(kind=kind, B=B, K=K, V=min(_vocab(rng), 128256), Hq=Hq, Hkv=Hkv, d=d, layers=min(layers, 4),
                    kv_lo=min(kv_lo, 16384), kv_hi=min(kv_hi, 16384), T=T, noise=noise, bf16=bf16, lens=lens)
    L_hi = rng.choice([4, 8, K])
    return dict(kind=kind, B=B, K=K, Hq=Hq, Hkv=Hkv, d=d, layers=layers, kv_lo=kv_lo, kv_hi=kv_hi, L_lo=0,
                L_hi=min(L_hi, K), tree=False, page=rng.choice([0, 0, 64, 128, 256]), lse=rng.random() < 0.3,
                lens=lens)


# ---------------------------------------------------------------------------------------------- lengths
def _kv(case):
    """Cache length of every sequence before the block: log-uniform in [kv_lo, kv_hi]."""
    r = np.random.default_rng([case["lens"], 1])
    lo, hi = math.log(case["kv_lo"]), math.log(case["kv_hi"])
    return np.clip(np.exp(r.uniform(lo, hi, case["B"])).round(), case["kv_lo"], case["kv_hi"]).astype(np.int32)


def _L(case):
    """Verified length of every sequence: uniform in [L_lo, L_hi]."""
    r = np.random.default_rng([case["lens"], 2])
    return r.integers(case["L_lo"], case["L_hi"] + 1, case["B"]).astype(np.int32)


def _temps(case):
    """One temperature for all, or greedy and sampling sequences in turn."""
    t = np.full(case["B"], case["T"], np.float32)
    if case.get("mixed"):
        t[::2] = 0.0
    return t


def _parents(case):
    return workloads.draft_tree(case["B"], case["K"], _L(case) if "L_lo" in case else case["K"], case["lens"] % 10007,
                                "ddtree", depth=24)


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _dtype(case):
    return torch.bfloat16 if case["bf16"] else torch.float32


def _logits(case, g):
    """Target logits N(0, 4^2) and a drafter that is the target plus noise; drafted tokens are the drafter's
    argmax (greedy sequences) or draws from its softmax (sampling ones)."""
    B, K, V, dt = case["B"], case["K"], case["V"], _dtype(case)
    target = torch.empty((B, K + 1, V), dtype=dt, device="cuda")
    draft = torch.empty((B, K, V), dtype=dt, device="cuda")
    tokens = torch.empty((B, K), dtype=torch.int32, device="cuda")
    temps = _temps(case)
    for b in range(B):
        x = torch.randn((K + 1, V), generator=g, device="cuda") * 4.0
        y = x[:K] + torch.randn((K, V), generator=g, device="cuda") * case["noise"]
        target[b], draft[b] = x.to(dt), y.to(dt)
        z = draft[b].float()
        if temps[b] > 0:
            u = torch.rand((K, V), generator=g, device="cuda").clamp_(1e-30, 1.0 - 1e-7)
            z = z / float(temps[b]) - torch.log(-torch.log(u))
        tokens[b] = torch.argmax(z, dim=-1).to(torch.int32)
    return target, draft, tokens, torch.from_numpy(temps).cuda()


def _cost(K):
    """Verification cost per length, convex and increasing, as the workloads' polynomial tables are."""
    t = np.arange(K + 1, dtype=np.float32)
    return torch.from_numpy((1.0 + 0.015 * t + 0.0005 * t * t).astype(np.float32)).cuda()


def _layers(case, g, kv, T):
    """Per layer Q [B,T,Hq,d] and a KV cache of N(0, 1) bf16, dense or in shuffled pages, with output buffers."""
    B, Hq, Hkv, d, page = case["B"], case["Hq"], case["Hkv"], case["d"], case.get("page", 0)
    need = int(kv.max()) + T
    bf = dict(dtype=torch.bfloat16, device="cuda")
    layers, table = [], None
    S = (need + 63) // 64 * 64
    if page:
        per = (need + page - 1) // page
        n_pages = B * per + 3
        table = torch.randperm(n_pages, generator=g, device="cuda")[:B * per].view(B, per).to(torch.int32).contiguous()
    for _ in range(case["layers"]):
        lay = {"Q": torch.randn((B, T, Hq, d), generator=g, **bf)}
        shape = (n_pages, Hkv, page, d) if page else (B, Hkv, S, d)
        for name in ("Kp", "Vp") if page else ("Kc", "Vc"):
            lay[name] = torch.randn(shape, generator=g, **bf)
        lay["O"] = torch.zeros_like(lay["Q"])
        if case.get("lse"):
            lay["lse"] = torch.zeros((B, T, Hq), dtype=torch.float32, device="cuda")
        layers.append(lay)
    return layers, table, (table.shape[1] * page if page else S)


def _dstat64(draft, tokens, temps):
    """(conf, row max, Z) of the drafter rows, in 64 bits."""
    conf, mx, Z = [], [], []
    for b in range(draft.shape[0]):
        x = draft[b].double()
        T = float(temps[b]) if float(temps[b]) > 0 else 1.0
        m = x.amax(dim=-1)
        e = torch.exp((x - m[:, None]) / T)
        z = e.sum(dim=-1)
        conf.append(e.gather(1, tokens[b].long()[:, None])[:, 0] / z)
        mx.append(m)
        Z.append(z)
    return torch.stack(conf), torch.stack([torch.stack(mx), torch.stack(Z)], dim=-1)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"kind": kind, "seed": int(seed)}
    if kind == "lm_head":
        M, V, Dm = case["M"], case["V"], case["Dm"]
        s["H"] = torch.randn((M, Dm), generator=g, device="cuda").to(torch.bfloat16)
        s["W"] = (torch.randn((V, Dm), generator=g, device="cuda") * (4.0 / Dm ** 0.5)).to(torch.bfloat16)
        s["tokens"] = torch.randint(0, V, (M,), generator=g, device="cuda").to(torch.int32)
        n_seq = (M + case["rows_per_seq"] - 1) // case["rows_per_seq"]
        s["temperature"] = torch.full((n_seq,), case["T"], dtype=torch.float32, device="cuda")
        s["rows_per_seq"] = case["rows_per_seq"]
        s["ws"] = lr.LmHeadWorkspace(M, V)
        return s
    B, K = case["B"], case["K"]
    if kind == "attn":
        kv = _kv(case)
        s["layers"], s["table"], S = _layers(case, g, kv, K + 1)
        s["kv_len"], s["L"] = torch.from_numpy(kv).cuda(), torch.from_numpy(_L(case)).cuda()
        s["parent"] = torch.from_numpy(_parents(case)).cuda() if case["tree"] else None
        s["lse"] = case["lse"]
        s["ws"] = lr.Workspace(B, K, 1, case["Hq"], case["Hkv"], case["d"], S)
        return s
    if kind == "accept_tree":
        V = case["V"]
        par = _parents(case)
        # siblings carry distinct tokens; each node's row favours the token of its first child (4 times in 5)
        tok = torch.stack([torch.randperm(V, generator=g, device="cuda")[:K] for _ in range(B)]).to(torch.int32)
        first = np.zeros((B, K + 1), np.int64)
        for b in range(B):
            for t in range(K, 0, -1):
                first[b, par[b, t]] = t
        x = torch.randn((B, K + 1, V), generator=g, device="cuda") * 4.0
        kid = torch.from_numpy(first).cuda()
        follow = (kid > 0) & (torch.rand((B, K + 1), generator=g, device="cuda") < 0.8)
        peak = torch.where(follow, tok.long().gather(1, (kid - 1).clamp_(min=0)),
                           torch.randint(0, V, (B, K + 1), generator=g, device="cuda"))
        x.scatter_add_(2, peak[:, :, None], torch.full((B, K + 1, 1), 12.0, device="cuda"))
        s["target"], s["tokens"], s["parent"] = x.to(_dtype(case)), tok.contiguous(), torch.from_numpy(par).cuda()
        s["L"] = torch.full((B,), K, dtype=torch.int32, device="cuda")
        s["temperature"] = torch.from_numpy(_temps(case)).cuda()
        s["ws"] = lr.Workspace(B, K, V)
        return s
    s["target"], s["draft"], s["tokens"], s["temperature"] = _logits(case, g)
    if kind == "accept":
        conf, dstat = _dstat64(s["draft"], s["tokens"], _temps(case))
        s["conf"], s["dstat"] = conf.float().contiguous(), dstat.float().contiguous()
        s["L"] = torch.from_numpy(_L(case)).cuda()
        s["ws"] = lr.Workspace(B, K, case["V"])
        return s
    s["cost"] = _cost(K)
    if kind == "select":
        del s["target"]
        s["ws"] = lr.Workspace(B, K, case["V"])
        return s
    kv = _kv(case)
    s["layers"], _, S = _layers(case, g, kv, K + 1)
    s["kv_len"] = torch.from_numpy(kv).cuda()
    s["ws"] = lr.Workspace(B, K, case["V"], case["Hq"], case["Hkv"], case["d"], S)
    return s


def run(state):
    s = state
    kind = s["kind"]
    if kind == "select":
        conf, dstat, L = lr.libraspec_confidence_select(s["draft"], s["tokens"], s["temperature"], s["cost"], s["ws"])
        return {"conf": conf, "dstat": dstat, "L": L}
    if kind == "attn":
        if s["table"] is None and s["parent"] is None:
            O, lse = lr.libraspec_verify_attn_layers(s["layers"], s["kv_len"], s["L"], s["ws"], want_lse=s["lse"])
        elif s["table"] is None:
            O, lse = lr.libraspec_verify_attn_tree_layers(s["layers"], s["parent"], s["kv_len"], s["L"], s["ws"],
                                                          want_lse=s["lse"])
        elif s["parent"] is None:
            O, lse = lr.libraspec_verify_attn_paged_layers(s["layers"], s["table"], s["kv_len"], s["L"], s["ws"],
                                                           want_lse=s["lse"])
        else:
            O, lse = lr.libraspec_verify_attn_tree_paged_layers(s["layers"], s["parent"], s["table"], s["kv_len"],
                                                                s["L"], s["ws"], want_lse=s["lse"])
        return {"O": O, "lse": lse}
    if kind == "accept":
        n, bonus = lr.libraspec_accept(s["target"], s["draft"], s["tokens"], s["conf"], s["dstat"], s["L"],
                                       s["temperature"], s["seed"], s["ws"], round_offset=1)
        return {"n_accepted": n, "bonus": bonus}
    if kind == "accept_tree":
        n, last, bonus = lr.libraspec_accept_tree(s["target"], s["tokens"], s["parent"], s["L"], s["temperature"],
                                                  s["seed"], s["ws"], round_offset=1)
        return {"n_accepted": n, "last": last, "bonus": bonus}
    if kind == "lm_head":
        stat, arg, prob = lr.libraspec_lm_head_stats(s["H"], s["W"], s["ws"], temperature=s["temperature"],
                                                     rows_per_seq=s["rows_per_seq"], tokens=s["tokens"])
        return {"max": stat[:, 0], "Z": stat[:, 1], "argmax": arg, "prob": prob}
    out = lr.libraspec_verify_round(s["draft"], s["tokens"], s["temperature"], s["cost"], s["target"], s["layers"],
                                    s["kv_len"], s["seed"], s["ws"], round_offset=1)
    return {"conf": out.conf, "dstat": out.dstat, "L": out.L, "n_accepted": out.n_accepted, "bonus": out.bonus_token,
            "O": out.O}


# ---------------------------------------------------------------------------------------------- the work
def _attn_work(case, kv, L):
    keys, rows = kv.astype(np.float64) + L + 1, L.astype(np.float64) + 1
    if case.get("tree"):  # a node sees the cache and its root path
        seen = np.zeros(case["B"])
        par = _parents(case)
        for b in range(case["B"]):
            depth = np.zeros(case["K"] + 1)
            for t in range(1, int(L[b]) + 1):
                depth[t] = depth[par[b, t]] + 1
            seen[b] = float(np.sum(kv[b] + 1 + depth[:int(L[b]) + 1]))
    else:
        seen = rows * kv + rows * (rows + 1) / 2
    b = case["Hkv"] * keys * case["d"] * 4 + rows * case["Hq"] * (case["d"] * 4 + (4 if case.get("lse") else 0))
    return case["layers"] * float(b.sum()), case["layers"] * float((case["Hq"] * seen * 4 * case["d"]).sum())


def _accept_bytes(case, L):
    """Rows a decision needs: a greedy sequence its L + 1, a sampling one its L and the row drawn from."""
    return float(np.sum(L + 1)) * case["V"] * (2 if case["bf16"] else 4)


def work(case):
    kind = case["kind"]
    eb = 2 if case.get("bf16") else 4
    if kind == "lm_head":
        M, V, Dm = case["M"], case["V"], case["Dm"]
        return {"bytes": (V + M) * Dm * 2 + M * 20, "flops": 2.0 * M * V * Dm}
    if kind == "select":
        return {"bytes": case["B"] * case["K"] * case["V"] * eb, "flops": 0}
    if kind == "attn":
        b, f = _attn_work(case, _kv(case), _L(case))
        return {"bytes": b, "flops": f}
    if kind == "accept":
        return {"bytes": _accept_bytes(case, _L(case)), "flops": 0}
    if kind == "accept_tree":
        return {"bytes": case["B"] * (case["K"] + 1) * case["V"] * eb, "flops": 0}
    L = np.full(case["B"], min(2, case["K"]))  # the lengths these drafters and cost tables select are short
    b, f = _attn_work(case, _kv(case), L)
    return {"bytes": b + case["B"] * case["K"] * case["V"] * eb + _accept_bytes(case, L), "flops": f}


def tolerance(case):
    kind = case["kind"]
    if kind in ("accept", "accept_tree"):
        return "exact"
    if kind == "select":
        # 32-bit sums and exponentials
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    if kind == "lm_head":
        # four times the distance from 64 bits (fp32 sums of 4096 products on the tensor cores, then exp)
        return {"rel": 1.2e-4, "max": 1e-3, "differ": 0.01}
    # bf16 probabilities and bf16 outputs: four times the distance from 64 bits (0.0023, single values 0.04)
    return {"rel": 1e-2, "max": 0.16, "differ": 0.01}


# ------------------------------------------------------------------------------------- the same in 64 bits
def _attn64(case, s, kv, L):
    """O and lse of every layer (zeros where nothing is verified)."""
    Hq, Hkv, d, T = case["Hq"], case["Hkv"], case["d"], case["K"] + 1
    g = Hq // Hkv
    par = _parents(case) if case.get("tree") else None
    Os, lses = [], []
    for lay in s["layers"]:
        O = torch.zeros((case["B"], T, Hq, d), dtype=torch.float64, device="cuda")
        lse = torch.zeros((case["B"], T, Hq), dtype=torch.float64, device="cuda")
        for b in range(case["B"]):
            n, rows = int(kv[b]) + int(L[b]) + 1, int(L[b]) + 1
            see = torch.zeros((rows, rows), dtype=torch.bool)
            for t in range(rows):
                if par is None:
                    see[t, :t + 1] = True
                else:
                    see[t, t] = True
                    see[t] |= see[int(par[b, t])] if t else see[t]
            hide = torch.zeros((rows, n), dtype=torch.bool)
            hide[:, int(kv[b]):] = ~see
            hide = hide.cuda()
            for h in range(Hkv):
                if s.get("table") is not None:
                    ids = s["table"][b].long()
                    k = lay["Kp"][ids, h].reshape(-1, d)[:n].double()
                    v = lay["Vp"][ids, h].reshape(-1, d)[:n].double()
                else:
                    k, v = lay["Kc"][b, h, :n].double(), lay["Vc"][b, h, :n].double()
                q = lay["Q"][b, :rows, h * g:(h + 1) * g].double()
                x = torch.einsum("thd,nd->thn", q, k) * d ** -0.5
                x.masked_fill_(hide[:, None, :], -math.inf)
                lse[b, :rows, h * g:(h + 1) * g] = torch.logsumexp(x, dim=-1)
                O[b, :rows, h * g:(h + 1) * g] = torch.einsum("thn,nd->thd", torch.softmax(x, dim=-1), v)
        Os.append(O)
        lses.append(lse)
    return Os, lses


def _select64(conf, cost):
    """The first length at which one more draft does not pay."""
    out = []
    for q in conf.cpu().numpy():
        P, E, n = 1.0, 1.0, 0
        while n < len(q):
            P *= float(q[n])
            if not P * float(cost[n]) > (float(cost[n + 1]) - float(cost[n])) * E:
                break
            E += P
            n += 1
        out.append(n)
    return np.array(out, np.int32)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("accept", "accept_tree"):
        return None  # whole numbers alone
    s = prepare(case, seed)
    if kind == "lm_head":
        M = case["M"]
        x = torch.empty((M, case["V"]), dtype=torch.float64, device="cuda")
        H = s["H"].double()
        for v in range(0, case["V"], 16384):
            x[:, v:v + 16384] = H @ s["W"][v:v + 16384].double().T
        m = x.amax(dim=-1)
        T = case["T"] if case["T"] > 0 else 1.0
        tok = x.gather(1, s["tokens"].long()[:, None])[:, 0]
        Z = torch.exp_((x - m[:, None]) / T).sum(dim=-1)
        return {"max": m, "Z": Z, "argmax": None, "prob": torch.exp((tok - m) / T) / Z}
    if kind == "attn":
        O, lse = _attn64(case, s, _kv(case), _L(case))
        return {"O": O, "lse": lse if case["lse"] else None}
    conf, dstat = _dstat64(s["draft"], s["tokens"], _temps(case))
    if kind == "select":
        return {"conf": conf, "dstat": dstat, "L": None}
    kv = _kv(case)
    O, _ = _attn64(case, s, kv, _select64(conf.float().double(), s["cost"].cpu().numpy()))
    return {"conf": conf, "dstat": dstat, "L": None, "n_accepted": None, "bonus": None, "O": O}
