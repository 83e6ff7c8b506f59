"""What the head is asked to do in use, as sized calls through its public entry points (`binding.MtpcHead`).

Four kinds of work, over the sizes the repository's workloads, tests and benchmark span:
  eval    log-likelihood of observed windows: the joint (`mtpc_window_logprob`), every prefix marginal
          (`mtpc_window_prefix_logprob`) or the loss value (`mtpc_window_loss`)
  train   one training step of the head: the loss over overlapping windows and all its gradients
          (`mtpc_window_loss_backward`, on a factored head `mtpc_lowrank_window_loss_backward`)
  decode  one speculative step of up to 128 sequences: draft windows with their prefix marginals
          (`mtpc_draft_sample_prefix`), then the acceptance stage against the target model's rows
          (`mtpc_speculative_accept`)
  batch   the same for a whole batch of positions at once, one window each
A case names the circuit family, the window length n, the width r, the vocabulary v (of which `symbols` exist), the
hidden size d, the dtype of the tensors handed in, and the adaptors' rank (0: one composed weight tensor). Inputs are
synthetic: hidden states ~N(0,1), weights ~N(0, 0.02), Zipf-distributed bytes, uniforms in [0,1).
"""
from __future__ import annotations

import math

import torch

from paper_2511_11346_b200 import binding

CP, HMM, HMM_CTX, BTREE = "cp", "hmm", "hmm_ctx", "btree"
FAMILY = {CP: binding.MTPC_CP, HMM: binding.MTPC_HMM, HMM_CTX: binding.MTPC_HMM, BTREE: binding.MTPC_BTREE}
GAMMA = 0.9              # discount of the training loss over the slots of a window


def _case(kind, family, n, r, v, d, *, seqs=0, length=0, out="joint", positions=0, wpp=1, symbols=0, dtype="bf16", rank=0):
    return {"kind": kind, "family": family, "n": n, "r": r, "v": v, "symbols": symbols or v, "d": d, "dtype": dtype,
            "rank": rank, "seqs": seqs, "length": length, "out": out, "positions": positions, "wpp": wpp}


def listed():
    return [
        # scoring a few short texts with a small mixture head: the smallest call, launches and host time count
        dict(_case("eval", CP, 4, 8, 256, 256, seqs=4, length=64, dtype="f32"), name="eval_cp_tiny"),
        # one sequence being decoded, one window per step: the latency of a speculative step
        dict(_case("decode", CP, 8, 16, 320, 4096, positions=1, wpp=1), name="decode_cp_1"),
        # a small serving batch, sixteen candidate windows each, the widest HMM head
        dict(_case("decode", HMM, 16, 32, 320, 4096, positions=8, wpp=16), name="decode_hmm_8"),
        # a large serving batch on a mixture head
        dict(_case("decode", CP, 16, 16, 320, 4096, positions=64, wpp=16), name="decode_cp_64"),
        # an uneven number of sequences on a tree head, a few windows each
        dict(_case("decode", BTREE, 8, 32, 256, 3072, positions=27, wpp=4), name="decode_btree_27"),
        # decoding with shared unembeddings and low-rank adaptors kept factored
        dict(_case("decode", CP, 8, 16, 320, 4096, positions=8, wpp=4, rank=16), name="decode_factored_8"),
        # log-likelihood of a training-sized batch: the benchmark's headline call
        dict(_case("eval", CP, 8, 16, 320, 4096, seqs=8, length=1024), name="eval_cp_8192"),
        # validation of an uneven batch of short texts, per-byte losses from a contextual HMM
        dict(_case("eval", HMM_CTX, 8, 32, 320, 4096, seqs=3, length=231, out="prefix"), name="eval_hmmctx_693"),
        # a training step on fp32 tensors of a padded vocabulary (268 symbols), uneven batch
        dict(_case("train", CP, 8, 16, 272, 3072, seqs=5, length=401, symbols=268, dtype="f32"), name="train_cp_f32_2005"),
        # a full training step of the tree head
        dict(_case("train", BTREE, 16, 32, 256, 3072, seqs=4, length=1024), name="train_btree_4096"),
        # a full training step with factored unembeddings
        dict(_case("train", HMM, 8, 32, 320, 4096, seqs=8, length=1024, rank=16), name="train_factored_8192"),
        # drafting and verifying a whole batch of positions, one window each
        dict(_case("batch", BTREE, 16, 32, 256, 3072, positions=4096, wpp=1), name="batch_btree_4096"),
    ]


# Multiply-adds of the projection in the largest drawn case of a kind, so that none costs more than the largest listed.
_MOST = {"eval": 2.8e12, "train": 1.6e12, "batch": 1.6e12}


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case of the same ranges: any family and dtype, every vocabulary, odd batch sizes."""
    kind = rng.choice(["eval", "train", "decode", "batch"])
    family = rng.choice([CP, CP, HMM, HMM_CTX, BTREE])
    n, r = rng.choice([4, 8, 16]), rng.choice([8, 16, 32])
    v, symbols = rng.choice([(256, 256), (272, 268), (320, 320)])
    d = rng.choice([1024, 2048, 3072, 4096])
    rank = rng.choice([0, 0, 0, 16, 32])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"]) if rank == 0 else "bf16"
    if kind == "decode":
        return _case(kind, family, n, r, v, d, positions=_log_uniform(rng, 1, 128), wpp=rng.choice([1, 4, 16]),
                     symbols=symbols, dtype=dtype, rank=rank)
    if kind == "batch" and v == 272:
        v, symbols = 320, 320                       # drafts of a padded vocabulary are verified up to 128 positions only
    positions = _log_uniform(rng, 200, 8192)
    positions = max(200, min(positions, int(_MOST[kind] / (n * r * v * d))))
    if kind == "batch":
        return _case(kind, family, n, r, v, d, positions=positions, wpp=1, symbols=symbols, dtype=dtype, rank=rank)
    seqs = rng.randint(1, 8)
    return _case(kind, family, n, r, v, d, seqs=seqs, length=positions // seqs, out=rng.choice(["joint", "prefix", "loss"]) if
                 kind == "eval" else "joint", symbols=symbols, dtype=dtype, rank=rank)


def _sum_units(case):
    """Sum units S whose r weights come from the hidden state."""
    n, r = case["n"], case["r"]
    return {CP: 1, HMM: 1, HMM_CTX: 1 + (n - 1) * r, BTREE: 1 + (n - 2) * r}[case["family"]]


def _positions(case):
    return case["positions"] or case["seqs"] * case["length"]


def _windows_of_text(case, g):
    """targets [T, n]: the n bytes after every position of `seqs` texts of Zipf-distributed bytes; -1 past a text's end."""
    n, seqs, length, symbols = case["n"], case["seqs"], case["length"], case["symbols"]
    rank_weight = 1.0 / torch.arange(1, symbols + 1, device="cuda", dtype=torch.float32) ** 1.1
    order = torch.randperm(symbols, device="cuda", generator=g)
    text = order[torch.multinomial(rank_weight, seqs * length, replacement=True, generator=g)].view(seqs, length)
    text = torch.cat([text, torch.full((seqs, n), -1, device="cuda")], dim=1).to(torch.int32)
    return text[:, 1:].unfold(1, n, 1)[:, :length].reshape(seqs * length, n).contiguous()


class _State:
    pass


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, r, v, d, rank, wpp = (case[k] for k in ("n", "r", "v", "d", "rank", "wpp"))
    T, f32 = _positions(case), torch.float32
    io = f32 if case["dtype"] == "f32" else torch.bfloat16

    def normal(*shape, std=1.0, dtype=io):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)

    def empty(*shape, dtype=f32):
        return torch.empty(shape, dtype=dtype, device="cuda")

    s = _State()
    s.case, s.T = case, T
    s.hidden = normal(T, d)
    W_sum = normal(_sum_units(case) * r, d, std=0.02)
    trans = None
    if case["family"] == HMM:
        trans = normal(n - 1, r, r, dtype=f32)
    elif case["family"] == HMM_CTX:                # the bias: a noisy identity, as after training from that start
        trans = normal(n - 1, r, r, dtype=f32) + 4.0 * torch.eye(r, device="cuda")
    W_emit = lowrank = None
    if rank:
        lowrank = (normal(n, v, d, std=0.02), normal(n, r, v, rank, std=0.05), normal(n, r, rank, d, std=0.05))
    else:
        W_emit = normal(n, r, v, d, std=0.02)
    s.head = binding.MtpcHead(FAMILY[case["family"]], n, r, v, d, binding.MTPC_F32 if io == f32 else binding.MTPC_BF16, T, wpp,
                              W_emit, W_sum, trans,
                              flags=binding.MTPC_FLAG_HMM_CONTEXTUAL if case["family"] == HMM_CTX else 0,
                              v_valid=case["symbols"] if case["symbols"] != v else 0, lowrank=lowrank)
    if case["kind"] in ("eval", "train"):
        s.targets = _windows_of_text(case, g)
        s.slot_loss, s.loss = empty(n), empty(1)
    if case["kind"] == "eval":
        s.out = empty(T, n) if case["out"] == "prefix" else empty(T)
    elif case["kind"] == "train":
        s.grads = {"hidden": empty(T, d), "W_sum": empty(*W_sum.shape)}
        if case["family"] == HMM:
            s.grads["T_static"] = empty(n - 1, r, r)
        if rank:
            s.grads.update(W_base=empty(n, v, d), A=empty(n, r, v, rank), B=empty(n, r, rank, d))
        else:
            s.grads["W_emit"] = empty(n, r, v, d)
    else:
        W = T * wpp
        s.uniforms = torch.rand(W, 2 * n, device="cuda", generator=g)
        s.accept_uniforms = torch.rand(W, n + 1, device="cuda", generator=g)
        # the target model's rows along the draft: flat enough that accepted lengths spread over the window, as they do
        # with a trained draft head; padding symbols have no mass
        logits = normal(W, n + 1, v, std=0.5, dtype=f32)
        logits[..., case["symbols"]:] = -math.inf
        s.target_probs = torch.softmax(logits, dim=-1)
        s.bytes, s.prefix = empty(W, n, dtype=torch.int32), empty(W, n)
        s.accepted, s.next_byte = empty(W, dtype=torch.int32), empty(W, dtype=torch.int32)
    return s


def run(s):
    case, head = s.case, s.head
    if case["kind"] == "eval":
        if case["out"] == "joint":
            head.mtpc_window_logprob(s.hidden, s.targets, s.out)
        elif case["out"] == "prefix":
            head.mtpc_window_prefix_logprob(s.hidden, s.targets, s.out)
        else:
            head.mtpc_window_loss(s.hidden, s.targets, case["seqs"], case["length"], GAMMA, s.slot_loss, s.loss)
            return {"slot_loss": s.slot_loss, "loss": s.loss}
        return s.out
    if case["kind"] == "train":
        gr = s.grads
        if case["rank"]:
            head.mtpc_lowrank_window_loss_backward(s.hidden, s.targets, case["seqs"], case["length"], GAMMA, s.slot_loss, s.loss,
                                                   gr["hidden"], gr["W_base"], gr["A"], gr["B"], gr["W_sum"],
                                                   gr.get("T_static"))
        else:
            head.mtpc_window_loss_backward(s.hidden, s.targets, case["seqs"], case["length"], GAMMA, s.slot_loss, s.loss,
                                           gr["hidden"], gr["W_emit"], gr["W_sum"], gr.get("T_static"))
        return {"slot_loss": s.slot_loss, "loss": s.loss, "grads": gr}
    head.mtpc_draft_sample_prefix(s.hidden, case["wpp"], s.uniforms, s.bytes, s.prefix)
    head.mtpc_speculative_accept(s.T, case["wpp"], s.bytes, s.prefix, s.target_probs, s.accept_uniforms, s.accepted, s.next_byte)
    return {"bytes": s.bytes, "prefix": s.prefix, "accepted": s.accepted, "next_byte": s.next_byte}


def work(case):
    """One pass: the weights, hidden states, targets or uniforms read once, the outputs written once; the projection of the
    hidden states onto every row (training: that contraction and its two gradients). Of the target model's rows the
    acceptance stage needs one value per drafted byte and one whole row per window."""
    n, r, v, d, rank = (case[k] for k in ("n", "r", "v", "d", "rank"))
    T, W, S = _positions(case), _positions(case) * case["wpp"], _sum_units(case) * r
    elt = 4 if case["dtype"] == "f32" else 2
    weights = (n * v * d + n * r * rank * (v + d) if rank else n * r * v * d) + S * d
    flops = 2.0 * T * (d * (n * v + n * r * rank + S) + n * r * v * rank if rank else d * (n * r * v + S))
    nbytes = elt * (weights + T * d)
    if case["kind"] == "eval":
        nbytes += 4 * T * n + 4 * (T * n if case["out"] == "prefix" else T if case["out"] == "joint" else n + 1)
    elif case["kind"] == "train":
        flops *= 3
        nbytes += 4 * T * n + 4 * (weights + T * d)
    else:
        nbytes += 4 * W * (2 * n + n + 1 + n + v) + 4 * W * (2 * n + 2)
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    """About four times what the calls differ by from the same steps in fp64: 1.1e-6 for values (fp32 sums of bf16 products),
    2.3e-3 for gradients (they pass the tensor cores as bf16). Drafts agree to 5e-7 except where a uniform lies on a
    boundary of its distribution (2 of 16384 bytes): such a window is another window, so one in W may differ, with its
    prefix marginals."""
    if case["kind"] == "eval":
        return {"rel": 5e-6}
    if case["kind"] == "train":
        return {"rel": 1e-2}
    W = _positions(case) * case["wpp"]
    return {"rel": min(1e-2, 0.1 / math.sqrt(W)), "max": 0.5, "differ": min(1e-2, 2e-3 + 1.0 / W)}
