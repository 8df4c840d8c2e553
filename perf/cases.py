"""Performance cases of the verify path: what a serving loop runs once per decoding step.

One pass is one verify cycle of a stack of layers over one batch, through the public driver of the package
(`harness.VerifyEngine`): branch_state_build and tree_verify_attn per layer, then accept_and_refresh over all layers.
Before the cycle the batch's committed lengths are written into the caches, as a scheduler does for the batch it
has put together; so every pass works at the lengths the case states, however often it is called.

Fields of a case
  dtype              storage type: "bf16" (the product shape: 64 heads x 512, indexer 4 x 128) or "fp32" (16 heads x 128,
                     indexer 1 x 64: the numerics configuration)
  B, D, layers       sequences, draft-tree nodes per sequence (root included), layers of the stack
  L_min, L_max       committed prefix lengths, uniform in [L_min, L_max] per sequence, any remainder
  topk               compressed entries selected per node
  tree               "random" (a tree per sequence) or "chain" (linear drafts)
  p                  probability that a node's target token is one of its drafted children
  page_tokens        0: one slab per sequence; else a paged pool with pages of that many tokens
  deferred           the refresh schedule that folds the 128-token blocks at commit time
  graph              the cycle replayed from a CUDA graph the program captured once, or launched call by call
"""
import math

import numpy as np
import torch

from paper_2609_24698_b200 import binding, harness, synth, workload

# Tokens a sequence may still grow by.  Every sequence has a slot for the longest one, and workspace and grids are sized
# for it, as in a server that does not know what comes.
ROOM = 512


def _case(name, B, layers, L_min, L_max, D=8, dtype="bf16", topk=512, tree="random", p=0.7, page_tokens=0, deferred=False, graph=True):
    return {"name": name, "dtype": dtype, "B": B, "D": D, "layers": layers, "L_min": L_min, "L_max": L_max, "topk": topk, "tree": tree,
            "p": p, "page_tokens": page_tokens, "deferred": deferred, "graph": graph}


def listed():
    return [
        # the smallest call: one short fp32 sequence, called by a program that keeps no graph
        _case("fp32_one_1k_calls", 1, 1, 1024, 1024, D=5, dtype="fp32", topk=64, graph=False),
        # an fp32 batch of mixed lengths
        _case("fp32_b16_mixed", 16, 1, 256, 4096, dtype="fp32", topk=64),
        # one user, linear drafts, called without a graph
        _case("one_4k_chain_calls", 1, 1, 4096, 4096, tree="chain", graph=False),
        # one user, tree drafts
        _case("one_4k_tree", 1, 1, 4096, 4096),
        # one user on a stack of layers, smallest budget: launches and latency of the whole cycle
        _case("one_short_stack", 1, 8, 256, 2048, D=5),
        # a small batch on a stack, launched call by call, with the deferred refresh schedule
        _case("b16_short_stack_calls", 16, 8, 256, 2048, D=6, deferred=True, graph=False),
        # chat: a batch of widely differing lengths
        _case("b16_chat", 16, 1, 512, 8192, p=0.65),
        # math and code prompts at full batch: the benchmark's workload
        _case("b64_short_stack", 64, 8, 256, 2048),
        # the same batch later in its generation: most nodes have to rank their candidates
        _case("b64_grown_stack", 64, 8, 1024, 4096),
        # a serving engine's paged pool
        _case("b32_paged_stack", 32, 4, 256, 4096, page_tokens=128),
        # long documents
        _case("b4_128k", 4, 1, 131072, 131072, topk=2048, p=0.6),
        # one long document in a paged pool
        _case("one_64k_paged", 1, 1, 65536, 65536, topk=2048, p=0.6, page_tokens=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.2:
        hi = _log_int(rng, 300, 4500)
        c = _case("", _log_int(rng, 1, 16), 1, _log_int(rng, 200, hi), hi, D=rng.randint(5, 8), dtype="fp32", topk=64,
                  tree=rng.choice(["random", "chain"]), graph=rng.random() < 0.6)
    else:
        while True:
            B, layers, hi = _log_int(rng, 1, 64), rng.choice([1, 2, 4, 8]), _log_int(rng, 256, 131072)
            if B * layers * hi <= 64 * 8 * 2048:
                break
        long = hi > 32768
        c = _case("", B, layers, _log_int(rng, max(200, hi // 16), hi), hi, D=rng.randint(5, 8), topk=2048 if long else 512,
                  tree=rng.choice(["random", "random", "chain"]), p=round(rng.uniform(0.5, 0.8), 2), page_tokens=rng.choice([0, 0, 128]),
                  deferred=rng.random() < 0.25, graph=rng.random() < 0.7)
    del c["name"]
    return c


def _shape(case):
    if case["dtype"] == "fp32":
        return synth.Shape("fp32", case["B"], case["D"], 16, 128, 4, case["topk"], 1, 64, 128, 128)
    return synth.Shape("bf16", case["B"], case["D"], 64, 512, 4, case["topk"], 4, 128, 128, 128)


def _trees(case, seed):
    cfg = synth.Config("case", 200, _shape(case), layers=case["layers"], tree=case["tree"], p_lo=case["p"], p_hi=case["p"], seed=seed)
    parent, n_nodes = synth.trees(cfg)
    draft, target = synth.tokens(cfg, 0, parent, n_nodes)
    return parent, n_nodes, draft, target


class _State:
    pass


# What accept_and_refresh writes, besides its own results: kept for all layers in one tensor each.
_UPDATED = ("L", "csa_kv", "csa_ik", "hca_kv", "win_kv", "csa_mx", "csa_s", "csa_acc_kv", "csa_acc_ik", "hca_mx", "hca_s", "hca_acc_kv")


def prepare(case, seed):
    sh, layers = _shape(case), case["layers"]
    rng = np.random.default_rng(seed)
    lengths = rng.integers(case["L_min"], case["L_max"] + 1, size=sh.B)
    csa_caps, hca_caps = harness.capacities(sh, [case["L_max"]] * sh.B, ROOM)
    eng = harness.VerifyEngine(sh, layers, csa_caps, hca_caps, case["L_max"] + ROOM + sh.D,
                               flags=binding.FLAG_HCA_DEFERRED if case["deferred"] else 0, page_tokens=case["page_tokens"])
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(t, spread):
        t.normal_(0.0, spread, generator=gen)

    # the caches: spreads of pooled vectors (4 and 128 tokens to an entry), open blocks as after one token
    st = _State()
    st.updated = {}
    for name in _UPDATED:
        st.updated[name] = torch.stack([getattr(c, name) for c in eng.caches])
        for l, c in enumerate(eng.caches):
            setattr(c, name, st.updated[name][l])
    u, d, di = st.updated, sh.d, sh.di
    normal(u["csa_kv"], 0.65 / math.sqrt(d)); normal(u["csa_ik"], 0.65 / math.sqrt(di)); normal(u["hca_kv"], 0.13 / math.sqrt(d))
    normal(u["win_kv"], 1 / math.sqrt(d))
    normal(u["csa_acc_kv"], 1 / math.sqrt(d)); normal(u["csa_acc_ik"], 1 / math.sqrt(di)); normal(u["hca_acc_kv"], 1 / math.sqrt(d))
    normal(u["csa_mx"], 1.0); normal(u["hca_mx"], 1.0)
    u["csa_s"].fill_(1.0); u["hca_s"].fill_(1.0)
    st.lengths = torch.from_numpy(np.tile(lengths.astype(np.int32), (layers, 1))).cuda()
    u["L"].copy_(st.lengths)
    out = torch.stack(eng.out)
    eng.out = list(out)

    # one cycle's inputs
    inp = harness.InputSet.empty(sh, layers)
    for nd in inp.layers:
        for t in (nd.q, nd.kv, nd.c_csa, nd.c_hca):
            normal(t, 1 / math.sqrt(d))
        normal(nd.ikc, 1 / math.sqrt(di)); normal(nd.iq, 1 / math.sqrt(di))
        normal(nd.g_csa, 1.0); normal(nd.g_hca, 1.0)
        normal(nd.iw, 1 / math.sqrt(sh.HI)); nd.iw.abs_()
    parent, n_nodes, draft, target = _trees(case, seed)
    for t, a in ((inp.layers[0].parent, parent), (inp.layers[0].n_nodes, n_nodes), (inp.draft, draft), (inp.target, target)):
        t.copy_(torch.from_numpy(a))

    st.engine, st.inputs = eng, inp
    st.graph = eng.capture(inp) if case["graph"] else None
    st.result = {"out": out, "accept_len": eng.accept_len, "accept_path": eng.accept_path, "bonus": eng.bonus, "status": eng.status, **u}
    return st


def run(state):
    state.updated["L"].copy_(state.lengths)
    if state.graph is not None:
        state.graph.replay()
    else:
        state.engine.launch_cycle(state.inputs)
    return state.result


def work(case):
    sh = _shape(case)
    lengths = np.linspace(case["L_min"], case["L_max"], sh.B + 2)[1:-1].astype(np.int64)
    w = workload.algorithmic_work(sh, case["layers"], lengths, _trees(case, 0)[0])
    return {"bytes": w["full_bytes"], "flops": w["flops"]}


def tolerance(case):
    # fp32: sums of a few hundred terms.  bf16: inputs, weights and results carry 8 bits; an entry whose score ties with
    # the last selected one to within fp32 rounding may be exchanged for it.
    return {"rel": 1e-5} if case["dtype"] == "fp32" else {"rel": 1e-2, "max": 0.3}
