"""The work that programs built on this library give it: decoding, prefill, training steps and factor export, each
through the public entry points, over the sizes that the configurations, tests and benchmark of this repository use.

A case is a dict of plain values:

  kind      "decode"   one token for B * H states                        (sfda_step / sfda_step_fused)
            "prefill"  the chunkwise forward                             (sfda_forward / sfda_forward_fused)
            "long"     the forward of few, long sequences                (sfda_forward_two_level)
            "train"    the forward and the gradients of a loss on it     (sfda_forward, sfda_backward; with raw inputs
                       also sfda_frontend before and sfda_frontend_backward after)
            "factors"  the chunk factors Gamma, Y, M, W and the phases   (sfda_chunk_factors)
  B, T, H, d_k, d_v, chunk, dtype ("bf16" or "f32")
  raw       the inputs are those of the stable parameterisation
  state     a non-zero initial state (and, in training, a cotangent of the final one)
  im        the imaginary part of the outputs is wanted as well

Inputs have the distributions of ``workloads``: alpha = sigmoid(N(3, 1)), theta ~ U(-pi, pi), beta = sigmoid(N(0, 1)),
unit keys, q and v ~ N(0, 1), states ~ N(0, 0.02); long sequences remember: alpha ~ U(0.999, 1), quantised phases and
one write in twenty.
"""
import math

import torch

import paper_2607_11897_b200 as sfda

ALPHA_MIN, ALPHA_MAX, THETA_MAX, EPS = 0.0, 1.0, math.pi, 1e-6


def _case(kind, B, T, H, d_k, d_v, chunk, dtype, raw=False, state=False, im=False, name=None):
    c = dict(kind=kind, B=B, T=T, H=H, d_k=d_k, d_v=d_v, chunk=chunk, dtype=dtype, raw=raw, state=state, im=im)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one conversation decoding token by token: latency, not bandwidth
        _case("decode", 1, 1, 32, 128, 128, 64, "bf16", name="decode_one_sequence"),
        # a full serving batch, the decode configuration, on the logits a layer's projections produce
        _case("decode", 256, 1, 32, 128, 128, 64, "bf16", raw=True, im=True, name="decode_batch_256"),
        # the small fp32 reference configuration: unit tests, debugging, toy models
        _case("prefill", 1, 256, 2, 64, 64, 16, "f32", name="prefill_tiny_fp32"),
        # an fp32 model of ordinary size with a prompt of no round length
        _case("prefill", 2, 2001, 16, 128, 128, 64, "f32", state=True, name="prefill_fp32_ragged"),
        # the 4k training / prefill configuration
        _case("prefill", 4, 4096, 16, 128, 128, 64, "bf16", im=True, name="prefill_4k"),
        # a batch of short ragged prompts on raw inputs, state carried over from the turn before
        _case("prefill", 16, 575, 19, 128, 128, 64, "bf16", raw=True, state=True, name="prefill_short_ragged_raw"),
        # the headline configuration: large-batch prefill
        _case("prefill", 8, 8192, 32, 128, 128, 64, "bf16", state=True, im=True, name="prefill_headline"),
        # the long-context configuration: few sequences of 131072 tokens
        _case("long", 1, 131072, 16, 128, 128, 64, "bf16", im=True, name="long_context"),
        # fine-tuning a small fp32 model on ragged sequences, gradients down to the raw inputs
        _case("train", 2, 333, 4, 64, 64, 32, "f32", raw=True, state=True, name="train_small_fp32_raw"),
        # one training step of a layer at the 4k configuration
        _case("train", 4, 4096, 16, 128, 128, 64, "bf16", name="train_4k"),
        # the same at the headline configuration, the state carried between segments of a document
        _case("train", 8, 8192, 32, 128, 128, 64, "bf16", raw=True, state=True, name="train_headline"),
        # factor export for a scan over chunk summaries outside the library
        _case("factors", 4, 8192, 32, 128, 128, 64, "bf16", name="factors_8k"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["decode", "prefill", "prefill", "train", "train", "prefill", "long", "factors"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    d_k, d_v = (128, 128) if rng.random() < 0.75 else (rng.choice([64, 128]), rng.choice([64, 128]))
    raw, state, im = rng.random() < 0.4, rng.random() < 0.5, rng.random() < 0.4
    H = rng.choice([1, 2, 4, 7, 8, 12, 16, 19, 24, 32])
    if kind == "decode":
        return _case(kind, _log_uniform(rng, 1, 256), 1, H, d_k, d_v, 64, dtype, raw=raw, im=im)
    if kind == "long":
        T = 1024 * rng.choice([16, 32, 48, 64, 96, 128])
        return _case(kind, 1, T, rng.choice([1, 2, 4, 8, 12, 16]), 128, 128, 64, "bf16", state=state, im=im)
    chunk = rng.choice([64, 64, 64, 128] if dtype == "bf16" or kind == "factors" else [16, 32, 64, 64])
    # tokens times heads from 512 to the kind's largest; T from 64 to 16384, round or not
    most = {("prefill", "bf16"): 1 << 21, ("prefill", "f32"): 1 << 17, ("train", "bf16"): 1 << 21,
            ("train", "f32"): 1 << 17, ("factors", "bf16"): 1 << 20, ("factors", "f32"): 1 << 18}[kind, dtype]
    rows = _log_uniform(rng, 512, most)
    T = _log_uniform(rng, 64, min(16384, max(64, rows // H)))
    if rng.random() < 0.5:
        T = max(64, T // 64 * 64)
    B = max(1, min(64, rows // (T * H)))
    return _case(kind, B, T, H, d_k, d_v, chunk, dtype, raw=raw and kind != "factors", state=state and kind != "factors",
                 im=im and kind == "prefill")


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, *shape, std=1.0):
        x = torch.randn(*shape, device="cuda", generator=self.g)
        return x if std == 1.0 else x.mul_(std)

    def uniform(self, lo, hi, *shape):
        return torch.rand(*shape, device="cuda", generator=self.g).mul_(hi - lo).add_(lo)


def _tokens(case, lead, r, dt):
    """q, k, v, alpha (a_raw), theta (b_raw), beta (c_raw) with the leading dimensions `lead`."""
    d_k, d_v, m = case["d_k"], case["d_v"], case["d_k"] // 2
    q = r.normal(*lead, d_k).to(dt)
    k = r.normal(*lead, d_k)
    if case["raw"]:
        k = k.mul_(torch.exp(r.normal(*lead, 1, std=0.5))).to(dt)
        a, b, c = r.normal(*lead, m).add_(3.0), r.normal(*lead, m, std=1.5), r.normal(*lead)
    else:
        k = k.div_(k.norm(dim=-1, keepdim=True)).to(dt)
        if case["kind"] == "long":
            p = torch.tensor([2.0, 3.0, 5.0, 7.0], device="cuda")[r.uniform(0, 4, lead[-1], m).long().clamp_(max=3)]
            a = r.uniform(0.999, 1.0, *lead, m)
            b = torch.floor(r.uniform(0, 1, *lead, m) * p).minimum(p - 1).mul_(2 * math.pi).div_(p)
            b = torch.where(b > math.pi, b - 2 * math.pi, b)
            c = (r.uniform(0, 1, *lead) < 0.05).float()
        else:
            a = torch.sigmoid(r.normal(*lead, m).add_(3.0))
            b = r.uniform(-math.pi, math.pi, *lead, m)
            c = torch.sigmoid(r.normal(*lead))
    v = r.normal(*lead, d_v).to(dt)
    return q, k, v, a.contiguous(), b.contiguous(), c.contiguous()


def prepare(case, seed):
    B, T, H, d_k, d_v, kind = case["B"], case["T"], case["H"], case["d_k"], case["d_v"], case["kind"]
    m, dt = d_k // 2, torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    code = sfda.SFDA_BF16 if case["dtype"] == "bf16" else sfda.SFDA_F32
    r = _Draw(seed)
    lead = (B, H) if kind == "decode" else (B, T, H)
    s = dict(case=dict(case))
    s["q"], s["k"], s["v"], s["a"], s["b"], s["c"] = _tokens(case, lead, r, dt)
    new = lambda *shape, dtype=torch.float32: torch.empty(*shape, device="cuda", dtype=dtype)  # noqa: E731
    scratch = lambda n: torch.empty(n, device="cuda", dtype=torch.uint8) if n else None        # noqa: E731
    if kind == "factors":
        del s["q"], s["v"]
        C, NC = case["chunk"], sfda.sfda_plan(T, case["chunk"])[0]
        s["out"] = (new(B, H, NC, m, 2), new(B, H, NC, m, C, 2), new(B, H, NC, C, C, 2), new(B, H, NC, m, C, 2),
                    new(B, T, H, m, dtype=torch.int32))
        return s
    s["o"] = new(*lead, d_v, dtype=dt)
    s["o_im"] = new(*lead, d_v, dtype=dt) if case["im"] else None
    if kind == "decode":
        s["S"] = r.normal(B, H, d_k, d_v, std=0.02)
        return s
    s["S0"] = r.normal(B, H, d_k, d_v, std=0.02) if case["state"] else None
    s["S_T"] = new(B, H, d_k, d_v)
    sizes = (B, T, H, d_k, d_v, case["chunk"], code)
    if kind == "long":
        s["ws"] = scratch(sfda.sfda_forward_two_level_workspace_bytes(*sizes))
    elif kind == "prefill" and case["raw"]:
        s["ws"] = scratch(sfda.sfda_forward_fused_workspace_bytes(*sizes))
    else:
        s["ws"] = scratch(sfda.sfda_workspace_bytes(*sizes))
    if kind == "train":
        s["d_o"] = r.normal(B, T, H, d_v).to(dt)
        s["dS_T"] = r.normal(B, H, d_k, d_v) if case["state"] else None
        s["grads"] = [torch.empty_like(s[x]) for x in ("q", "k", "v", "a", "b", "c")] + [new(B, H, d_k, d_v)]
        if case["raw"]:
            s["param"] = [torch.empty_like(s[x]) for x in ("a", "b", "c", "k")]
        s["bws"] = scratch(sfda.sfda_backward_workspace_bytes(B, T, H, d_k, d_v, code))
    return s


def run(s):
    case = s["case"]
    kind, chunk = case["kind"], case["chunk"]
    q, k, v, a, b, c = (s.get(x) for x in ("q", "k", "v", "a", "b", "c"))
    scalars = (ALPHA_MIN, ALPHA_MAX, THETA_MAX, EPS)
    if kind == "factors":
        sfda.sfda_chunk_factors(k, a, b, c, *s["out"], chunk)
        return s["out"]
    if kind == "decode":
        if case["raw"]:
            sfda.sfda_step_fused(q, k, v, a, b, c, *scalars, s["S"], s["o"], s["o_im"])
        else:
            sfda.sfda_step(q, k, v, a, b, c, s["S"], s["o"], s["o_im"])
        return s["o"], s["o_im"], s["S"]
    if kind == "long":
        sfda.sfda_forward_two_level(q, k, v, a, b, c, s["S0"], s["o"], s["o_im"], s["S_T"], chunk, 0, s["ws"])
        return s["o"], s["o_im"], s["S_T"]
    if kind == "prefill":
        if case["raw"]:
            sfda.sfda_forward_fused(q, k, v, a, b, c, *scalars, s["S0"], s["o"], s["o_im"], s["S_T"], chunk, s["ws"])
        else:
            sfda.sfda_forward(q, k, v, a, b, c, s["S0"], s["o"], s["o_im"], s["S_T"], chunk, s["ws"])
        return s["o"], s["o_im"], s["S_T"]
    al, th, be, ku = a, b, c, k
    if case["raw"]:
        al, th, be, ku = s["param"]
        sfda.sfda_frontend(a, b, c, k, *scalars, al, th, be, ku)
    sfda.sfda_forward(q, ku, v, al, th, be, s["S0"], s["o"], s["o_im"], s["S_T"], chunk, s["ws"])
    dq, dk, dv, da, db, dc, dS0 = s["grads"]
    sfda.sfda_backward(q, ku, v, al, th, be, s["S0"], s["d_o"], None, s["dS_T"], dq, dk, dv, da, db, dc, dS0, s["bws"])
    if case["raw"]:
        sfda.sfda_frontend_backward(a, b, c, k, *scalars, da, db, dc, dk, da, db, dc, dk)
    return (s["o"], s["S_T"]) + tuple(s["grads"])


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def work(case):
    B, T, H, d_k, d_v, kind = case["B"], case["T"], case["H"], case["d_k"], case["d_v"], case["kind"]
    e, m, rows, states = 2 if case["dtype"] == "bf16" else 4, d_k // 2, B * T * H, B * H * d_k * d_v * 4
    keys = d_k * e + 2 * m * 4 + 4                       # k, alpha, theta, beta of a row
    inputs = keys + d_k * e + d_v * e
    outputs = d_v * e * (2 if case["im"] else 1)
    if kind == "decode":
        # per state: decay and rotate, k^* S, the rank-one update, S^* q: four complex multiply-adds per element
        return {"bytes": rows * (inputs + outputs) + 2 * states, "flops": rows * 4 * 8 * m * d_v}
    C = 64
    chunks = B * H * -(-T // C)
    if kind == "factors":
        C = case["chunk"]
        n = B * H * -(-T // C)
        return {"bytes": rows * (keys + 4 * m) + n * (8 * m + 16 * m * C + 8 * C * C), "flops": n * (4 * m * C * C + 4 * C ** 3 // 3)}
    # the chunkwise form with chunks of 64: two Gram matrices, the triangular system and the outputs' lower triangle,
    # three products with the state
    forward = chunks * (4 * d_k * C * C + 12 * C * d_k * d_v + 8 * C * C * d_v)
    total = {"bytes": rows * (inputs + outputs) + states * (2 if case["state"] else 1), "flops": forward}
    if kind == "train":
        # the adjoint reads the inputs and the cotangents once and writes a gradient for every input; it repeats the
        # forward's state products and has two for the cotangent of the state and three for the gradients of its own
        total["bytes"] += rows * (2 * inputs + d_v * e) + states * (3 if case["state"] else 1)
        total["flops"] += 2 * forward + chunks * 8 * C * d_k * d_v
        if case["raw"]:
            total["bytes"] += rows * 2 * keys
    return total


def tolerance(case):
    """Relative 2-norm.  bf16 forwards round every operand of the tensor-core products to bf16 (2^-9 each): 4.5e-3
    against 64-bit arithmetic, 5.1e-3 to 6.4e-3 with the two-level scan.  Everything else computes in fp32 (up to
    6e-7, sums in another order about twice that); bf16 outputs are rounded once (1.7e-3)."""
    kind, bf16 = case["kind"], case["dtype"] == "bf16"
    if kind == "long":
        return {"rel": 2.5e-2}
    if kind in ("prefill", "train") and bf16:
        return {"rel": 1.8e-2}
    if kind == "decode" and bf16:
        return {"rel": 7e-3}
    return {"rel": 5e-6}
