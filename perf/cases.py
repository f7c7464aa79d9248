"""The work that a program has this library do, as a list of cases that can be timed.

A case names an operation and its sizes:

  step       mtv_verify_step: heads, tree attention of every layer, acceptance on stored logits, compaction
  chain      mtv_verify_steps: consecutive steps in one call, each first writing its tree's K/V rows with the rotary
             embedding, the acceptance fed by the fused LM head
  host       mtv_verify_step_host: the step for a caller whose per-step tensors live in pinned host memory
  attention  tree_verify_attention, one call per layer, as a backbone calls it between its own layers
  heads      medusa_heads_topk alone (the drafting half of a step)
  lm_head    lm_head_argmax and tree_accept_keys (the verifying half, logits never stored)

Every state's inputs are made on the GPU from the seed alone: activations, queries, keys and values ~ N(0, 1), weights
~ N(0, 1) / sqrt(fan-in), base-model logits ~ N(0, 1) with a greedy walk planted down the tree (probability 0.3, 0.6
or 0.9 per level, by sequence), prefix lengths uniform in [lo, hi].
"""
import math
import random

import torch

from paper_2603_03383_b200 import binding

DEV = "cuda"
BF16 = torch.bfloat16


def _case(name, op, B=1, lo=0, hi=0, H=0, Hq=0, Hkv=0, D=128, V=0, K=4, tree="rank_prior", T=64, layers=32, spare=0, steps=1):
    """lo, hi: prefix lengths; tree: "rank_prior" (T nodes) or the top-k per depth of a full tree ("4,2,2"); spare: cache
    rows beyond those that the longest sequence needs (a serving cache is larger than what it holds at the moment)."""
    c = dict(op=op, B=B, lo=lo, hi=hi, H=H, Hq=Hq, Hkv=Hkv, D=D, V=V, K=K, tree=tree, T=T, layers=layers, spare=spare, steps=steps)
    return dict(c, name=name) if name else c


def listed():
    b7 = dict(H=4096, Hq=32, Hkv=8, V=131072)   # the 7B-class shape of the benchmark configurations
    return [
        # The five benchmark configurations as whole steps.  tiny: every kernel is latency, launches count.
        _case("step tiny", "step", lo=128, hi=128, H=512, Hq=8, Hkv=2, D=64, V=1024, K=3, tree="4,2,2", T=29),
        # A chat turn at the start: the heads' weight stream dominates, attention is short.
        _case("step short", "step", lo=512, hi=512, **b7),
        # The headline: one long sequence.
        _case("step long", "step", lo=8192, hi=8192, **b7),
        # A serving batch of unequal sequences.
        _case("step batched", "step", B=16, lo=1024, hi=4096, **b7),
        # Long contexts and the widest tree: attention dominates and is bound by the tensor cores.
        _case("step stress", "step", B=4, lo=32768, hi=32768, K=5, T=128, **b7),
        # Decoding without the host between the steps: two sequences, groups of seven query heads, a smaller vocabulary.
        _case("chain of two steps", "chain", B=2, lo=700, hi=3000, H=3584, Hq=28, Hkv=4, V=32000, spare=1000, steps=2),
        # The step end to end for a host program (queries and logits go up, attention outputs come down).
        _case("host step long", "host", lo=8192, hi=8192, **b7),
        # Layer-by-layer attention inside a backbone: one long sequence; a ragged batch in a roomy cache; small heads.
        _case("attention long", "attention", lo=8192, hi=8192, Hq=32, Hkv=8, layers=8),
        _case("attention ragged", "attention", B=7, lo=300, hi=6001, Hq=28, Hkv=4, layers=8, spare=2047),
        _case("attention head size 64", "attention", B=3, lo=97, hi=5003, Hq=16, Hkv=2, D=64, K=5, T=128, layers=8),
        # Drafting for a few sequences, a vocabulary that no tile divides.
        _case("heads five rows", "heads", B=5, H=4096, V=50003),
        # Verifying many nodes at once: the LM head becomes a dense contraction.
        _case("LM head 1024 nodes", "lm_head", B=8, H=4096, V=131072, K=5, T=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "chain", "host", "attention", "attention", "attention", "heads", "lm_head"])
    K = rng.choice([2, 3, 4, 4, 5])
    if rng.random() < 0.25:
        topk = [rng.randint(2, 4)] + [rng.randint(1, 2) for _ in range(min(K, 4) - 1)]
        K, tree, T, n = len(topk), ",".join(map(str, topk)), 1, 1
        for k in topk:
            n *= k
            T += n
    else:
        tree, T = "rank_prior", rng.randint(16, 128)
    D = 64 if rng.random() < 0.2 else 128
    Hkv, G = rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 3, 4, 4, 5, 6, 7, 8])
    Hq = Hkv * G
    V = _log_int(rng, 1000, 131072)
    H = 64 * _log_int(rng, 8, 64)
    B = _log_int(rng, 1, 16)
    hi = _log_int(rng, 64, 32768)
    layers = rng.randint(4, 32)
    if op in ("step", "chain", "host", "attention"):
        layers = layers if op != "attention" else 8
        row = 4 * B * Hkv * D * layers              # bytes of K and V that one more token of every sequence takes
        hi = max(64, min(hi, int((8e9 if op != "host" else 2e9) / row)))
    lo = hi if rng.random() < 0.3 else max(1, int(hi * rng.uniform(0.1, 1.0)))
    spare = rng.choice([0, 0, rng.randint(1, max(2, hi // 4))])
    c = dict(B=B, K=K, tree=tree, T=T)
    if op in ("heads", "lm_head"):
        return _case("", op, H=H, V=V, layers=1, **c)
    if op == "attention":
        return _case("", op, lo=lo, hi=hi, Hq=Hq, Hkv=Hkv, D=D, layers=layers, spare=spare, **c)
    steps = rng.randint(2, 3) if op == "chain" else 1
    return _case("", op, lo=lo, hi=hi, H=H, Hq=Hq, Hkv=Hkv, D=D, V=V, layers=layers, spare=spare, steps=steps, **c)


# ------------------------------------------------------------------------------------------------ inputs
class _Draws:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)
        self.py = random.Random(seed)

    def normal(self, *shape, scale=1.0):
        t = torch.empty(shape, dtype=BF16, device=DEV)
        flat = t.view(-1)
        for s in range(0, flat.numel(), 1 << 30):
            flat[s:s + (1 << 30)].normal_(0.0, scale, generator=self.g)
        return t

    def ints(self, lo, hi, *shape):
        return torch.randint(lo, hi + 1, shape, generator=self.g, device=DEV, dtype=torch.int32)


def _i32(*shape):
    return torch.zeros(shape, dtype=torch.int32, device=DEV)


def _tree(c):
    if c["tree"] == "rank_prior":
        return binding.Tree(c["K"], binding.tree_gen_rank_prior(c["K"], c["T"]))
    return binding.Tree(c["K"], binding.tree_gen_cartesian([int(k) for k in c["tree"].split(",")]))


def _candidates(tree, hidden, W1, b1, W2):
    """The tree's tokens as plain PyTorch finds them (fp32), to plant an acceptance on; the root's token is left at 0."""
    h, toks = hidden.float(), [torch.zeros(hidden.shape[0], 1, dtype=torch.int64, device=DEV)]
    for k in range(tree.K):
        x = h + torch.nn.functional.silu(h @ W1[k].float().T + b1[k].float())
        z = torch.cat([x @ w.float().T for w in W2[k].split(1 << 16)], dim=1)
        toks.append(z.topk(tree.k_d[k], dim=1).indices)
    return torch.cat(toks, dim=1)[:, tree.tree_indices]


def _plant(r, tree, B, V, tree_tok):
    """(sequence, node, token) of a greedy walk down the tree: where it goes on, the token is a child's, where it ends it
    is none's."""
    tok, at = tree_tok.tolist(), []
    children = [[j for j in range(1, tree.T) if tree.parent[j] == i] for i in range(tree.T)]
    for b in range(B):
        node, p = 0, (0.3, 0.6, 0.9)[b % 3] if B > 1 else 0.6
        while True:
            ch = children[node]
            if ch and r.py.random() < p:
                nxt = r.py.choices(ch, weights=[1.0 / (tree.rank[c] + 1) for c in ch])[0]
                at.append((b, node, tok[b][nxt]))
                node = nxt
                continue
            taken = {tok[b][c] for c in ch}
            at.append((b, node, next(t for t in range(V) if t not in taken)))
            break
    return torch.tensor(at, device=DEV).T


def _logits(r, tree, B, V, tree_tok):
    x = r.normal(B, tree.T, V)
    b, node, tok = _plant(r, tree, B, V, tree_tok)
    x[b, node, tok] = 16.0
    return x


def _final_hidden(r, tree, B, V, W_lm, tree_tok):
    """Hidden states whose most likely token is the planted one (any token at the nodes off the walk)."""
    tok = r.ints(0, V - 1, B, tree.T).long()
    b, node, t = _plant(r, tree, B, V, tree_tok)
    tok[b, node] = t
    H = W_lm.shape[1]
    return W_lm[tok] + r.normal(B, tree.T, H, scale=0.3 * H ** -0.5)


def _heads(r, c, s):
    B, H, V, K = c["B"], c["H"], c["V"], c["K"]
    s.update(W1=r.normal(K, H, H, scale=H ** -0.5), b1=r.normal(K, H, scale=0.1), W2=r.normal(K, V, H, scale=H ** -0.5))


def _draft(r, c, tree):
    B = c["B"]
    return dict(hidden=r.normal(B, c["H"]), root_tok=r.ints(0, c["V"] - 1, B), cand=_i32(B, tree.C),
                cand_logit=torch.zeros(B, tree.C - 1, device=DEV), tree_tok=_i32(B, tree.T))


def _accepted(c, tree):
    B, K1 = c["B"], tree.K + 1
    return dict(accept_len=_i32(B), best_path=_i32(B), acc_nodes=_i32(B, K1), acc_tok=_i32(B, K1), next_root=_i32(B))


def _caches(r, c, tree, s):
    B, n = c["B"], c["layers"]
    s["Lcap"] = c["hi"] + tree.T + (c["steps"] - 1) * (tree.K + 1) + c["spare"]
    s["K"] = r.normal(n, B, c["Hkv"], s["Lcap"], c["D"])
    s["V"] = r.normal(n, B, c["Hkv"], s["Lcap"], c["D"])
    s["lens0"] = r.ints(c["lo"], c["hi"], B)
    s["lens0"][-1] = c["hi"]
    s["lens"], s["status"] = s["lens0"].clone(), _i32(B)
    for x in "KV":
        s[x + "_ptrs_host"] = binding.cache_pointer_array(list(s[x]))
        s[x + "_ptrs"] = s[x + "_ptrs_host"].to(DEV)


def _step_args(c, tree, s, d):
    a = binding.StepArgs()
    for n in ("B", "H", "V", "Hq", "Hkv", "D"):
        setattr(a, n, c[n])
    a.n_layers, a.Lcap = c["layers"], s["Lcap"]
    a.stride_b, a.stride_h, a.stride_t = s["K"].stride()[1:4]
    fields = dict(d, W1=s["W1"], b1=s["b1"], W2=s["W2"], k_caches=s["K_ptrs"], v_caches=s["V_ptrs"],
                  k_caches_host=s["K_ptrs_host"], v_caches_host=s["V_ptrs_host"], seq_lens=s["lens"], status=s["status"], ws=s["ws"])
    for n, t in fields.items():
        if hasattr(a, n):
            setattr(a, n, t.data_ptr())
    a.ws_bytes = s["ws"].numel()
    return a


def prepare(case, seed):
    c, r = case, _Draws(seed)
    tree, op, B = _tree(c), c["op"], c["B"]
    s = dict(op=op, tree=tree, case=c)
    n = binding.mtv_workspace_bytes(tree, B, c["H"] or 8, c["V"] or 8, c["Hq"], c["Hkv"], c["D"], c["hi"] + tree.T + (c["steps"] - 1) * (tree.K + 1) + c["spare"])
    s["ws"] = torch.zeros(n, dtype=torch.uint8, device=DEV)
    if op == "lm_head":                 # the drafted tokens are an input here: distinct candidates
        cand = torch.stack([torch.randperm(c["V"], generator=r.g, device=DEV)[:tree.C] for _ in range(B)])
        tok = cand[:, tree.tree_indices]
        s["tree_tok"], s["out"] = tok.to(torch.int32).contiguous(), _accepted(c, tree)
        s["W_lm"] = r.normal(c["V"], c["H"], scale=c["H"] ** -0.5)
        s["x"] = _final_hidden(r, tree, B, c["V"], s["W_lm"], tok)
        s.update(keys=torch.zeros(B * tree.T, dtype=torch.int64, device=DEV), am=_i32(B, tree.T), am_val=torch.zeros(B, tree.T, device=DEV))
        s["outputs"] = [s["am"], s["am_val"], s["out"]]
        return s
    if op == "attention":
        _caches(r, c, tree, s)
        s["q"] = r.normal(c["layers"], B, tree.T, c["Hq"], c["D"])
        s["out"] = torch.zeros_like(s["q"])
        s["layers"] = list(zip(s["q"], s["K"], s["V"], s["out"]))
        s["outputs"] = [s["out"], s["status"]]
        return s
    _heads(r, c, s)
    if op == "heads":
        s.update(_draft(r, c, tree))
        s["outputs"] = [s["cand"], s["cand_logit"], s["tree_tok"]]
        return s
    _caches(r, c, tree, s)
    if op == "chain":
        s["W_lm"] = r.normal(c["V"], c["H"], scale=c["H"] ** -0.5)
    s["parts"], s["args"], s["appends"] = [], [], []
    for step in range(c["steps"]):
        d = dict(_draft(r, c, tree), **_accepted(c, tree))
        tok = _candidates(tree, d["hidden"], s["W1"], s["b1"], s["W2"])
        d["q_layers"] = r.normal(c["layers"], B, tree.T, c["Hq"], c["D"])
        d["out_layers"] = torch.zeros_like(d["q_layers"])
        if op == "chain":
            d["x_final"], d["W_lm"] = _final_hidden(r, tree, B, c["V"], s["W_lm"], tok), s["W_lm"]
            d["k_new"], d["v_new"] = (r.normal(c["layers"], B, tree.T, c["Hkv"], c["D"]) for _ in range(2))
            ap = binding.AppendArgs()
            ap.k_new_layers, ap.v_new_layers, ap.rope_theta = d["k_new"].data_ptr(), d["v_new"].data_ptr(), 0.0
            s["appends"].append(ap)
        else:
            d["logits"] = _logits(r, tree, B, c["V"], tok)
        a = _step_args(c, tree, s, d)
        if step:
            a.root_tok = None           # the previous step's next_root, on the device
        s["parts"].append(d)
        s["args"].append(a)
    names = ["cand", "cand_logit", "tree_tok", "out_layers", "accept_len", "best_path", "acc_nodes", "acc_tok", "next_root"]
    if op == "host":
        d, names = s["parts"][0], names[:2]
        up = {n: d[n].cpu().pin_memory() for n in ("hidden", "root_tok", "q_layers", "logits")}
        down = {n: torch.zeros(t.shape, dtype=t.dtype, pin_memory=True) for n, t in
                [(n, d[n]) for n in ("tree_tok", "out_layers", "accept_len", "best_path", "acc_nodes", "acc_tok", "next_root")] + [("seq_lens", s["lens"])]}
        s["host_in"], s["host_out"], s["host_args"] = up, down, binding.StepArgs()
        for n, t in list(up.items()) + list(down.items()):
            setattr(s["host_args"], n, t.data_ptr())
    # what the step leaves: its results, the lengths, and the caches (as a few whole tensors) that it writes into
    n = max(1, (1 << 30) // s["K"][0].numel())
    s["outputs"] = [[d[n] for n in names] for d in s["parts"]] + [s.get("host_out"), s["lens"], s["status"], [x for k in "KV" for x in s[k].split(n)]]
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    s = state
    op, tree = s["op"], s["tree"]
    if op == "attention":
        for q, k, v, out in s["layers"]:
            binding.tree_verify_attention(tree, q, k, v, s["lens"], out, s["ws"], status=s["status"])
    elif op == "heads":
        binding.medusa_heads_topk(tree, s["hidden"], s["W1"], s["b1"], s["W2"], s["root_tok"], s["cand"], s["cand_logit"], s["tree_tok"], s["ws"])
    elif op == "lm_head":
        o = s["out"]
        binding.lm_head_argmax(tree, s["x"], s["W_lm"], s["keys"], s["am"], s["am_val"])
        binding.tree_accept_keys(tree, s["case"]["B"], s["keys"], s["tree_tok"], o["accept_len"], o["best_path"], o["acc_nodes"], o["acc_tok"], o["next_root"])
    else:
        s["lens"].copy_(s["lens0"])     # a step advances the lengths on the device: each pass begins where the request begins
        if op == "host":
            binding.mtv_verify_step_host(tree, s["args"][0], s["host_args"])
        elif op == "chain":
            binding.mtv_verify_steps(tree, s["args"], s["appends"])
        else:
            binding.mtv_verify_step(tree, s["args"][0])
    return s["outputs"]


# ------------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    c = case
    T, B, n = c["T"], c["B"], c["steps"]
    mean = (c["lo"] + c["hi"]) / 2 + T
    by, fl = 0.0, 0.0
    if c["op"] in ("step", "chain", "host", "heads"):
        by += n * 2.0 * c["K"] * c["H"] * (c["H"] + c["V"] + 1)
        fl += n * 2.0 * B * c["K"] * c["H"] * (c["H"] + c["V"])
    if c["op"] in ("step", "chain", "host", "attention"):
        by += n * c["layers"] * B * (4.0 * mean * c["Hkv"] * c["D"] + 4.0 * T * c["Hq"] * c["D"])
        fl += n * c["layers"] * B * 4.0 * T * c["Hq"] * c["D"] * mean
    if c["op"] in ("chain", "lm_head"):
        by += n * 2.0 * (c["V"] * c["H"] + B * T * c["H"])
        fl += n * 2.0 * B * T * c["V"] * c["H"]
    if c["op"] == "chain":              # new K/V rows read and written, rotated queries written
        by += n * c["layers"] * B * T * (8.0 * c["Hkv"] * c["D"] + 2.0 * c["Hq"] * c["D"])
    if c["op"] in ("step", "host"):
        by += 2.0 * B * T * c["V"]
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # token ids, lengths, nodes and cache rows are whole values or copies: the same; bf16 attention outputs and fp32 sums
    # as their types give
    if case["op"] in ("heads", "lm_head"):
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.1}
