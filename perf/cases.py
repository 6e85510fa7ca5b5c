"""The work that users of this framework have it do, as cases that can be timed and compared.

A decoding loop of relaxed speculative decoding drafts tokens (``csd_sample_rows``, one call per draft
position), verifies them (``csd_verify``, ``csd_verify_ex``, or ``csd_verify_tree`` for static trees) and emits;
logits of an offline scorer may sit in host memory (``csd_verify_host``), and those of a tensor-parallel LM
head are slices of the vocabulary (``csd_verify_sharded``).  Shapes are those of the workloads this
repository configures and tests: image vocabularies of 4096 to 65536 tokens, 2 to 16 drafted positions, batches of 1
to 256 sequences, fp32 and bf16 logits, classifier-free guidance and top-k filtering.
"""
import math

import numpy as np
import torch

import paper_2601_09212_b200 as csd
from paper_2601_09212_b200 import workloads as W
from paper_2601_09212_b200.vocab_sharded import ShardedRound, csd_verify_sharded

_DEFAULTS = dict(entry="ex", B=1, gamma=8, V=16384, dtype="f32", rho=0.9, law="gauss", bonus=True, guidance=0.0, top_k=0,
                 overlapped=False)
TREE = (4, 3, 2, 2)   # candidates per level of the static draft tree
SHARDS = 4            # ranks of the tensor-parallel LM head


def _case(name, **kw):
    return dict(_DEFAULTS, **kw, **({"name": name} if name else {}))


def listed():
    guided = dict(dtype="bf16", guidance=4.0, top_k=1000)
    return [
        # one image at a time: the smallest call, where latency is everything; the simple entry point
        _case("chain_b1_f32", entry="simple", B=1, gamma=4, bonus=False),
        # a small serving batch on fp32 logits, with the bonus row
        _case("chain_b16_f32", B=16),
        # the headline workload (guidance mix, top-k) in a decoding loop: each call waits for the one before it
        _case("guided_b64_bf16", B=64, **guided),
        # the same for independent requests whose calls may overlap on the GPU
        _case("guided_b64_overlapped", B=64, overlapped=True, **guided),
        # few sequences over a large vocabulary with the filter that goes with it
        _case("guided_b4_v65536", B=4, V=65536, dtype="bf16", guidance=3.0, top_k=2000),
        # a large batch of long drafts with heavy-tailed bf16 logits
        _case("heavy_b256_bf16", B=256, gamma=16, dtype="bf16", law="student3", rho=0.85, bonus=False),
        # the largest: fp32 logits over a large vocabulary
        _case("wide_b256_f32", B=256, V=65536),
        # a vocabulary with a few special tokens added: rows of odd length, most of them not 16-byte aligned
        _case("odd_b24_bf16", B=24, gamma=7, V=16387, dtype="bf16"),
        # one draft position of a batch of 64: a token per row from the guided, filtered drafter
        _case("draft_r64_bf16", entry="draft", B=64, gamma=0, bonus=False, **guided),
        # a static draft tree, guided and filtered
        _case("tree_b16_bf16", entry="tree", B=16, gamma=0, bonus=False, **guided),
        # logits in pinned host memory: copies in, the round, copies out
        _case("host_b8_bf16", entry="host", B=8, **guided),
        # one rank's round on its quarter of the vocabulary
        _case("shard_b64_bf16", entry="shard", B=64, V=4096, dtype="bf16"),
    ]


def _rows(c):
    """Logit rows of one pass, per array."""
    if c["entry"] == "tree":
        return c["B"] * 2 * (sum(TREE) + 1)
    if c["entry"] == "draft":
        return c["B"]
    return c["B"] * (2 * c["gamma"] + int(c["bonus"]))


def _logit_bytes(c):
    return _rows(c) * c["V"] * (4 if c["dtype"] == "f32" else 2) * (2 if c["guidance"] else 1)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    entry = rng.choices(("ex", "simple", "draft", "tree", "host", "shard"), (55, 10, 10, 10, 5, 10))[0]
    while True:
        c = _case("", entry=entry, B=log_int(1, 256), gamma=rng.randint(2, 16), rho=round(rng.uniform(0.7, 0.97), 3))
        c["V"] = log_int(4096, 65536)
        c["law"] = rng.choice(("gauss", "gauss", "student3"))
        odd = entry == "ex" and rng.random() < 0.2
        if not odd:
            c["V"] = c["V"] // 8 * 8   # rows of whole 16-byte vectors
        if entry == "simple":
            c["bonus"] = False
        else:
            c["dtype"] = rng.choice(("f32", "bf16", "bf16"))
            c["bonus"] = rng.random() < 0.7
            if rng.random() < 0.5:
                c["guidance"] = round(rng.uniform(2.0, 7.5), 2)
            if entry != "shard" and rng.random() < (0.8 if c["guidance"] else 0.3):
                c["top_k"] = min(log_int(200, 2000), c["V"] // 8)
            c["overlapped"] = entry == "ex" and rng.random() < 0.3
        if entry in ("draft", "tree"):
            c["gamma"], c["bonus"] = 0, False
        if entry == "shard":
            c["V"] = max(1024, c["V"] // SHARDS // 8 * 8)
        # no dearer than the listed ones: host logits cross PCIe, and odd rows and trees cost more per byte
        most = {"host": 8e6, "tree": 8e7}.get(entry, (2e7 if c["top_k"] else 1e8) if odd else 1e9)
        if _logit_bytes(c) <= most:
            return c


def _workload(c, seed):
    kw = dict(B=c["B"], V=c["V"], dtype=W.F32 if c["dtype"] == "f32" else W.BF16, rho=c["rho"], law=c["law"], top_k=c["top_k"],
              cfg=c["guidance"] > 0, seed=seed, device="cuda")
    if c["guidance"]:
        kw["cfg_scale"] = c["guidance"]
    if c["entry"] == "tree":
        return W.make_tree(W.static_tree(TREE), schedule=csd.csd_make_schedule(1, 1.1, 0.7, len(TREE)), **kw)
    gamma = max(1, c["gamma"])
    return W.make("case", gamma=gamma, bonus_row=c["bonus"], schedule=csd.csd_make_schedule(1, 1.1, 0.7, gamma), **kw)


def _ints(*shape):
    return torch.empty(*shape, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    c = dict(case)
    w = _workload(c, seed)
    B, L = c["B"], c["gamma"]
    st = dict(entry=c["entry"], w=w)
    if c["entry"] == "simple":
        st["out"] = (_ints(B, L + 1), _ints(B))
    elif c["entry"] == "draft":
        rows = w.draft_logits[:, 0].contiguous()
        st.update(rows=rows, uncond=None if w.draft_uncond is None else w.draft_uncond[:, 0].contiguous(),
                  u=w.uniforms[:, 0].contiguous(), out=(_ints(B), _ints(B)),
                  ws=torch.zeros(csd.csd_sample_workspace_size(B, c["V"], w.dtype), dtype=torch.uint8, device="cuda"))
        st["w"] = dict(cfg_scale=w.cfg_scale, top_k=w.top_k)
    elif c["entry"] == "tree":
        D = len(TREE)
        st.update(out=(_ints(B, D + 1), _ints(B), _ints(B, D), _ints(B)),
                  ws=torch.zeros(csd.csd_tree_workspace_size(B, w.N, w.V, w.dtype), dtype=torch.uint8, device="cuda"))
    elif c["entry"] == "shard":
        pqf = torch.empty(3, B, L, device="cuda")
        st.update(out=(_ints(B, L + 1), _ints(B), _ints(B), pqf),
                  round=ShardedRound(w.target_logits, w.draft_logits, w.draft_tokens, w.uniforms, w.relax_schedule, v_offset=0,
                                     V_total=SHARDS * c["V"], shard=0, n_shards=SHARDS, target_uncond=w.target_uncond,
                                     draft_uncond=w.draft_uncond, cfg_scale=w.cfg_scale))
    elif c["entry"] == "host":
        host = {k: None if getattr(w, k) is None else getattr(w, k).cpu().pin_memory()
                for k in ("target_logits", "draft_logits", "target_uncond", "draft_uncond", "draft_tokens", "uniforms",
                          "relax_schedule")}
        out = tuple(torch.zeros(n, dtype=torch.int32).pin_memory() for n in ((B, L + 1), (B,), (B,)))
        prm = csd.make_params(host["target_logits"], host["draft_logits"], host["draft_tokens"], host["uniforms"],
                              host["relax_schedule"], out[0], out[1], target_uncond=host["target_uncond"],
                              draft_uncond=host["draft_uncond"], cfg_scale=w.cfg_scale, top_k=w.top_k, out_status=out[2], host=True)
        st.update(w=host, out=out, prm=prm,
                  staging=torch.empty(csd.csd_host_staging_size(prm), dtype=torch.uint8, device="cuda"))
    else:
        pqf = torch.empty(3, B, L, device="cuda")   # P and Q at the drafted tokens and the acceptance probabilities
        out = (_ints(B, L + 1), _ints(B), _ints(B), pqf)
        ws = csd.new_workspace(B, L, c["V"], w.dtype)
        prm = csd.make_params(w.target_logits, w.draft_logits, w.draft_tokens, w.uniforms, w.relax_schedule, out[0], out[1],
                              target_uncond=w.target_uncond, draft_uncond=w.draft_uncond, cfg_scale=w.cfg_scale, top_k=w.top_k,
                              out_status=out[2], dbg_p=pqf[0], dbg_q=pqf[1], dbg_f=pqf[2], workspace=ws,
                              back_to_back=c["overlapped"])
        st.update(out=out, ws=ws, prm=prm)
    return st


def _gather(t):
    """Stands in for the all-gather of a few KB between the ranks: every rank reports this rank's numbers."""
    return t.expand(SHARDS, *t.shape).contiguous()


def run(st):
    w, out, entry = st["w"], st["out"], st["entry"]
    if entry == "ex":
        csd.csd_verify_ex(st["prm"])
    elif entry == "simple":
        csd.csd_verify(w.target_logits, w.draft_logits, w.draft_tokens, w.uniforms, w.relax_schedule, out[0], out[1])
    elif entry == "draft":
        csd.csd_sample_rows(st["rows"], st["u"], out[0], uncond=st["uncond"], cfg_scale=w["cfg_scale"], top_k=w["top_k"],
                            out_status=out[1], workspace=st["ws"])
    elif entry == "tree":
        csd.csd_verify_tree(w.target_logits, w.draft_logits, w.parent, w.draft_tokens, w.uniforms, w.relax_schedule, out[0],
                            out[1], target_uncond=w.target_uncond, draft_uncond=w.draft_uncond, cfg_scale=w.cfg_scale,
                            top_k=w.top_k, out_nodes=out[2], out_status=out[3], workspace=st["ws"])
    elif entry == "shard":
        csd_verify_sharded(st["round"], out[0], out[1], out[2], gather=_gather, dbg_p=out[3][0], dbg_q=out[3][1], dbg_f=out[3][2])
    else:
        csd.csd_verify_host(st["prm"], st["staging"])
    return out


def work(case):
    c = dict(case)
    B, L = c["B"], c["gamma"]
    if c["entry"] == "tree":
        n, d = sum(TREE), len(TREE)
        small = B * (4 * n + 4 * (n + 1) + 4 * (d + 1) + 4 * d + 8) + 4 * d
    elif c["entry"] == "draft":
        small = B * 12
    else:
        small = B * (4 * L + 4 * (L + 1) * 2 + 8) + 4 * L
        if c["entry"] in ("ex", "shard"):
            small += B * L * 12
    # per logit: an exponential, its argument and a sum (and the mix)
    return {"bytes": _logit_bytes(c) + small, "flops": _rows(c) * c["V"] * (7 if c["guidance"] else 4)}


def tolerance(case):
    # Probabilities are fp32 arithmetic on identical inputs whatever the storage type: against a softmax in
    # 64 bits p, q and f were seen to differ by up to 1.4e-7 (relative, 2-norm) and 7e-7 (largest).  A token or
    # accepted length differs only where a uniform lies within a rounding error of an accept threshold or a
    # boundary of the CDF: 0 to 3 sequences in a thousand, of which a small batch holds at most one.
    return {"rel": 6e-7, "max": 3e-6, "differ": 0.01}
