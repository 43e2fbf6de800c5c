"""The work that is timed and compared when the library is tuned: calls that a program built on it makes, through the
public entry points, over the range of sizes they are meant for.

Kinds of case
  step       photon_decode_step: append, coarse attention, converter, chunk attention, everything on the device
  step_host  photon_decode_step_host: the same step for a serving loop whose inputs and results are host buffers
  advance    one meta-context boundary of recursive generation (Section 2.3.3, steps i-iii) through one layer a level:
             context chunker (photon_rmsnorm, photon_linear) -> photon_encoder_step -> photon_converter ->
             photon_decoder_prefill over the fresh prefix vectors
  decoder    photon_decoder_step: one layer of the local decoders for the newest position of every in-flight chunk
  prefill    photon_decoder_prefill alone: one layer over the prefix vectors of n chunks
  teacher    photon_chunk_causal_attn over whole chunks, the form a teacher-forced pass has

Model shapes are those of the library's workloads (16/4 heads x 128 at width 2048, 8/8 x 128 at 1024, 4/2 x 64 at 256).
All tensors are bf16, the one data type of the library.  Values: activations, queries, keys and values N(0,1), weights
N(0, 1/fan-in), scales of the normalisations around one.  A serving program keeps the lengths of its sequences itself
and hands them in with a step, which is also what lets a pass be repeated on the same state: the step starts by
writing the lengths it is told (a chunk boundary empties the chunk buffers the same way).
"""
from __future__ import annotations

import torch

import paper_2512_20687_b200 as ph

BF16 = torch.bfloat16
MODELS = {  # name: Hq, Hkv, dh, P, C
    "tiny": (4, 2, 64, 4, 4),
    "1b": (16, 4, 128, 4, 4),
    "wide": (8, 8, 128, 8, 16),
}
PAGE = 64        # rows per page of a paged coarse cache


def _case(kind, model, n, **kw):
    """n: sequences (step, step_host, advance) or in-flight chunks (decoder, prefill, teacher)."""
    c = {"kind": kind, "model": model, "n": n, "S": 0, "per_seq": 0, "ragged": False, "paged": False, "shared": 0,
         "lse": False, "bias": False, "out_major": False}
    c.update(kw)
    return c


def listed():
    c = []
    # The smallest call there is: two short sequences of the tiny model.  Latency and launches are all of it.
    c.append(dict(_case("step", "tiny", 2, S=16, per_seq=8), name="step_tiny"))
    # Interactive serving of a 1B-class model: 64 sequences of 8192 tokens, two chunks of each in flight.
    c.append(dict(_case("step", "1b", 64, S=512, per_seq=2, out_major=True), name="step_1b"))
    # Continuous batching: an odd number of sequences of all ages in a paged cache, log-sum-exp and bias asked for.
    c.append(dict(_case("step", "1b", 77, S=1000, per_seq=2, ragged=True, paged=True, lse=True, bias=True), name="step_ragged_paged"))
    # Few sequences with a long context (131072 tokens).
    c.append(dict(_case("step", "1b", 16, S=8192, per_seq=2, out_major=True), name="step_long"))
    # Many queries against one document: 256 branches behind a shared prefix of 2048 latents.
    c.append(dict(_case("step", "1b", 256, S=32, per_seq=2, shared=2048, out_major=True), name="step_shared"))
    # Throughput serving, all chunks of 512 sequences decoded in parallel: the largest call in bytes.
    c.append(dict(_case("step", "wide", 512, S=128, per_seq=32), name="step_chunks"))
    # The interactive step fed from host memory, results back on the host.
    c.append(dict(_case("step_host", "1b", 64, S=512, per_seq=2, out_major=True), name="step_host_1b"))
    # The top-level stream moves on by one latent and every sequence gets a fresh chunk to decode.
    c.append(dict(_case("advance", "1b", 64, S=512, ragged=True, out_major=True), name="advance_1b"))
    # A token for each of a small number of in-flight chunks: the weights are most of what is read.
    c.append(dict(_case("decoder", "1b", 127), name="decoder_1b"))
    # A token for each of 16384 in-flight chunks: the tensor cores' case.
    c.append(dict(_case("decoder", "wide", 16384), name="decoder_chunks"))
    # Prefix pass over an odd number of fresh chunks: over a thousand rows, between the two cases above.
    c.append(dict(_case("prefill", "1b", 301, out_major=True), name="prefill_1b"))
    # Teacher-forced attention over whole chunks, most of them complete.
    c.append(dict(_case("teacher", "wide", 16384), name="teacher_chunks"))
    return c


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    while True:
        kind = rng.choice(("step", "step", "step", "step_host", "advance", "decoder", "decoder", "prefill", "teacher"))
        model = rng.choice(("1b", "1b", "wide", "tiny"))
        if kind in ("step", "step_host", "advance"):
            c = _case(kind, model, _log_int(rng, 1, 512), S=_log_int(rng, 16, 8192), ragged=rng.random() < 0.6,
                      out_major=rng.random() < 0.5)
            if kind != "advance":
                c["per_seq"] = rng.choice((2, 2, 8, 32))
                c["lse"], c["bias"] = rng.random() < 0.3, rng.random() < 0.3
            if kind == "step" and rng.random() < 0.25:
                c["shared"], c["S"] = _log_int(rng, 128, 4096), _log_int(rng, 8, 256)
            elif rng.random() < 0.3:
                c["paged"] = True
        else:
            c = _case(kind, model, _log_int(rng, 1, 16384 if kind != "prefill" else 2048))
            c["out_major"] = kind != "teacher" and rng.random() < 0.5
        w = work(c)
        if w["bytes"] <= 8e8 and w["flops"] <= 3.5e11:
            return c


def _shape(case):
    Hq, Hkv, dh, P, C = MODELS[case["model"]]
    D = Hq * dh
    return Hq, Hkv, dh, P, C, D, max(64, round(2.75 * D / 64) * 64)


# ---- inputs ------------------------------------------------------------------------------------------------------------


class _Context:
    """A library context that goes with the state that uses it."""

    def __init__(self, Hq, Hkv, dh, D, P, C, max_queries):
        self.h = ph.photon_create(Hq, Hkv, dh, D, P, C, max_queries)

    def __del__(self):
        if torch is not None and torch.cuda is not None:                        # (not while the interpreter shuts down)
            torch.cuda.synchronize()
            ph.photon_destroy(self.h)


class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator("cuda").manual_seed(int(seed))

    def normal(self, *shape, std=1.0):
        t = torch.empty(*shape, dtype=BF16, device="cuda").normal_(generator=self.g)
        return t if std == 1.0 else t.mul_(std)

    def scales(self, n):
        return torch.empty(n, device="cuda").normal_(1.0, 0.1, generator=self.g).to(BF16)

    def ints(self, n, lo, hi):
        return torch.randint(lo, hi + 1, (n,), generator=self.g, device="cuda", dtype=torch.int32)

    def linear(self, k, n, out_major):
        return self.normal(n, k, std=k ** -0.5) if out_major else self.normal(k, n, std=k ** -0.5)


def _coarse_lengths(case, d):
    """Rows per sequence before the step: S - 1 each, or of all ages."""
    n, S = case["n"], case["S"]
    return d.ints(n, 0, S - 1) if case["ragged"] else torch.full((n,), S - 1, dtype=torch.int32, device="cuda")


def _coarse(case, d, s, shared=True):
    Hq, Hkv, dh, _, _, _, _ = _shape(case)
    n, S = case["n"], case["S"]
    s["len0"] = _coarse_lengths(case, d)
    s["len"] = s["len0"].clone()
    kw = {}
    if case["paged"]:
        pages = -(-S // PAGE)
        s["k"], s["v"] = d.normal(n * pages, Hkv, PAGE, dh), d.normal(n * pages, Hkv, PAGE, dh)
        s["table"] = torch.randperm(n * pages, generator=d.g, device="cuda").to(torch.int32).view(n, pages).contiguous()
        kw["page_table"] = s["table"]
    else:
        s["k"], s["v"] = d.normal(n, Hkv, S, dh), d.normal(n, Hkv, S, dh)
    if case["shared"] and shared:
        L = case["shared"]
        kw.update(k_shared=d.normal(1, Hkv, L, dh), v_shared=d.normal(1, Hkv, L, dh),
                  shared_len=torch.full((1,), L, dtype=torch.int32, device="cuda"),
                  shared_id=torch.zeros(n, dtype=torch.int32, device="cuda"))
    s["kv"] = ph.make_kv(s["k"], s["v"], s["len"], max_len=S, **kw)


def _chunks(case, d, s, n, lengths):
    _, Hkv, dh, P, C, _, _ = _shape(case)
    s["clen0"] = lengths
    s["clen"] = lengths.clone()
    s["kc"], s["vc"] = d.normal(n, Hkv, P + C, dh), d.normal(n, Hkv, P + C, dh)
    s["ckv"] = ph.make_kv(s["kc"], s["vc"], s["clen"])


def _layer(case, d):
    Hq, Hkv, dh, _, _, D, F = _shape(case)
    om = case["out_major"]
    return ph.make_layer(d.scales(D), d.linear(D, (Hq + 2 * Hkv) * dh, om), d.linear(D, D, om), d.scales(D),
                         d.linear(D, 2 * F, om), d.linear(F, D, om), int(om), F)


def _step_state(case, d, s):
    Hq, Hkv, dh, P, C, D, _ = _shape(case)
    n, Nc = case["n"], case["n"] * case["per_seq"]
    s["ctx"] = _Context(Hq, Hkv, dh, D, P, C, max(n, Nc))
    _coarse(case, d, s)
    _chunks(case, d, s, Nc, d.ints(Nc, P + 1, P + C))
    inputs = [d.normal(n, Hkv, dh), d.normal(n, Hkv, dh), d.normal(n, Hq, dh), s["len0"], d.normal(Nc, Hq, dh)]
    outputs = [torch.empty(n, Hq, dh, dtype=BF16, device="cuda"), torch.empty(Nc, Hq, dh, dtype=BF16, device="cuda")]
    if case["lse"]:
        outputs.insert(1, torch.empty(n, Hq, device="cuda"))
    s["w"] = d.linear(D, P * D, case["out_major"])
    s["bias"] = d.normal(P * D, std=0.1) if case["bias"] else None
    s["U"] = torch.empty(n, P, D, dtype=BF16, device="cuda")
    if case["kind"] == "step_host":
        # one page-locked buffer each way; what the chunk attention reads and writes comes last
        dev_in, at_in = _pack(inputs)
        dev_out, at_out = _pack(outputs)
        host_in, s["host_out"] = dev_in.cpu().pin_memory(), torch.empty(dev_out.numel(), dtype=torch.uint8).pin_memory()
        inputs = [_view(dev_in, o, t) for o, t in zip(at_in, inputs)]
        s["host_views"] = [_view(s["host_out"], o, t) for o, t in zip(at_out, outputs)]
        outputs = [_view(dev_out, o, t) for o, t in zip(at_out, outputs)]
        s["len"] = inputs[3]
        s["kv"].len = s["len"].data_ptr()
        s["io"] = ph.HostIO(host_in, dev_in, dev_out, s["host_out"], in_split=at_in[4], out_split=at_out[-1])
    k_new, v_new, q, _, q_chunk = inputs
    s["k_new"], s["v_new"], s["q"], s["q_chunk"] = k_new, v_new, q, q_chunk
    s["out"], s["lse"], s["out_chunk"] = outputs[0], outputs[1] if case["lse"] else None, outputs[-1]
    s["args"] = ph.make_step_args(s["kv"], k_new, v_new, q, s["out"], dh ** -0.5, s["w"], int(case["out_major"]), s["U"], n,
                                  chunks=s["ckv"], q_chunk=q_chunk, out_chunk=s["out_chunk"], Nc=Nc, scale_chunk=dh ** -0.5,
                                  bias=s["bias"], lse_coarse=s["lse"])


def _pack(tensors):
    at, end = [], 0
    for t in tensors:
        at.append(end)
        end += -(-t.numel() * t.element_size() // 256) * 256
    buf = torch.zeros(end, dtype=torch.uint8, device="cuda")
    for o, t in zip(at, tensors):
        _view(buf, o, t).copy_(t)
    return buf, at


def _view(buf, at, like):
    return buf[at:at + like.numel() * like.element_size()].view(like.dtype).view(like.shape)


def _advance_state(case, d, s):
    Hq, Hkv, dh, P, C, D, F = _shape(case)
    n, om = case["n"], case["out_major"]
    s["ctx"] = _Context(Hq, Hkv, dh, D, P, C, n)
    _coarse(case, d, s)
    _chunks(case, d, s, n, torch.zeros(n, dtype=torch.int32, device="cuda"))
    s["latents"], s["gamma"] = d.normal(n, 4 * D), d.scales(4 * D)             # four lower-level latents per sequence
    s["w_chunker"], s["b_chunker"] = d.linear(4 * D, D, om), d.normal(D, std=0.1)
    s["encoder"], s["w"], s["decoder"] = _layer(case, d), d.linear(D, P * D, om), _layer(case, d)
    new = lambda *shape: torch.empty(*shape, dtype=BF16, device="cuda")
    s["normed"], s["a"], s["x"], s["U"], s["y"] = new(n, 4 * D), new(n, D), new(n, D), new(n, P, D), new(n, P, D)
    s["scratch"] = ph.make_layer_scratch(n * P, Hq, Hkv, dh, F, "cuda", BF16)


def prepare(case, seed):
    Hq, Hkv, dh, P, C, D, F = _shape(case)
    n, kind, d, s = case["n"], case["kind"], _Draw(seed), {}
    s["kind"], s["scale"], s["layout"] = kind, dh ** -0.5, int(case["out_major"])
    if kind in ("step", "step_host"):
        _step_state(case, d, s)
    elif kind == "advance":
        _advance_state(case, d, s)
    else:
        s["ctx"] = _Context(Hq, Hkv, dh, D, P, C, n)
        if kind == "decoder":
            _chunks(case, d, s, n, d.ints(n, P, P + C - 1))
            s["x"], rows = d.normal(n, D), n
        elif kind == "prefill":
            _chunks(case, d, s, n, torch.zeros(n, dtype=torch.int32, device="cuda"))
            s["x"], rows = d.normal(n, P, D), n * P
        else:
            # three chunks in four are complete, the rest end somewhere behind the prefix
            part = d.ints(n, P + 1, P + C)
            _chunks(case, d, s, n, torch.where(d.ints(n, 0, 3) == 0, part, torch.full_like(part, P + C)))
            s["x"] = d.normal(n, P + C, Hq, dh)
        s["y"] = torch.empty_like(s["x"])
        if kind != "teacher":
            s["layer"] = _layer(case, d)
            s["scratch"] = ph.make_layer_scratch(rows, Hq, Hkv, dh, F, "cuda", BF16)
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------------


def run(s):
    kind, ctx, scale = s["kind"], s["ctx"].h, s["scale"]
    if kind == "step":
        s["len"].copy_(s["len0"])
        ph.photon_decode_step(ctx, s["args"])
        return [s["out"], s["lse"], s["U"], s["out_chunk"], s["len"], s["k"], s["v"]]
    if kind == "step_host":                                                     # the lengths come with the host buffer
        ph.photon_decode_step_host(ctx, s["args"], s["io"])
        return [s["host_views"], s["U"], s["len"], s["k"], s["v"]]
    if kind == "advance":
        s["len"].copy_(s["len0"])
        ph.photon_rmsnorm(ctx, s["latents"], s["gamma"], 1e-5, s["normed"])
        ph.photon_linear(ctx, s["normed"], s["w_chunker"], s["layout"], s["b_chunker"], s["a"])
        ph.photon_encoder_step(ctx, s["encoder"], s["scratch"], s["a"], s["kv"], s["x"], scale=scale)
        ph.photon_converter(ctx, s["x"], s["w"], s["layout"], None, s["U"])
        s["clen"].zero_()
        ph.photon_decoder_prefill(ctx, s["decoder"], s["scratch"], s["U"], s["ckv"], None, s["y"], scale=scale)
        return [s["a"], s["x"], s["U"], s["y"], s["len"], s["k"], s["v"], s["clen"], s["kc"], s["vc"]]
    if kind == "decoder":
        s["clen"].copy_(s["clen0"])
        ph.photon_decoder_step(ctx, s["layer"], s["scratch"], s["x"], s["ckv"], s["y"], scale=scale)
        return [s["y"], s["clen"], s["kc"], s["vc"]]
    if kind == "prefill":
        s["clen"].zero_()
        ph.photon_decoder_prefill(ctx, s["layer"], s["scratch"], s["x"], s["ckv"], None, s["y"], scale=scale)
        return [s["y"], s["clen"], s["kc"], s["vc"]]
    ph.photon_chunk_causal_attn(ctx, s["ckv"], s["x"], None, s["y"], scale=scale)
    return [s["y"]]


# ---- what a pass cannot do without -------------------------------------------------------------------------------------


def work(case):
    """Bytes: weights, valid key and value rows, inputs and outputs once each; no intermediate of a layer.  Flops: the
    contractions.  Lengths that are drawn count with their means."""
    Hq, Hkv, dh, P, C, D, F = _shape(case)
    n, kind = case["n"], case["kind"]
    row = Hkv * dh * 4                                                          # a key and a value row, all heads
    layer_w = D * (Hq + 2 * Hkv) * dh + D * D + 3 * D * F
    rows_c = (case["S"] + 1) / 2 if case["ragged"] else case["S"]
    coarse = (n * rows_c + case["shared"]) * row
    coarse_f = n * (rows_c + case["shared"]) * Hq * dh * 4
    if kind in ("step", "step_host"):
        Nc, rows = n * case["per_seq"], P + (C + 1) / 2
        return {"bytes": coarse + 2 * n * row + D * P * D * 2 + n * P * D * 2 + Nc * rows * row + 4 * (n + Nc) * D,
                "flops": coarse_f + 2 * n * D * P * D + Nc * rows * Hq * dh * 4}
    if kind == "advance":
        return {"bytes": coarse + 2 * n * row + 2 * (2 * layer_w + 4 * D * D + P * D * D) + 2 * n * D * (4 + 3 + 3 * P) + n * P * row,
                "flops": 2 * n * (layer_w * (1 + P) + 4 * D * D + P * D * D) + coarse_f}
    if kind == "teacher":
        rows = P + C - (C - 1) / 8
        return {"bytes": n * rows * row + n * (P + C) * D * 4, "flops": n * Hq * dh * 2 * rows * (rows + 1)}
    rows = n * P if kind == "prefill" else n
    kv = n * row * (P if kind == "prefill" else P + (C + 1) / 2 + 1)
    return {"bytes": 2 * layer_w + 4 * rows * D + kv, "flops": 2 * rows * layer_w}


def tolerance(case):
    """Four times the error against the same path in 64 bits without a rounding in between, as measured on these cases
    (2-norm; largest difference over the rms or the value): a bf16 output has 1.7e-3 to 2.8e-3 and 1.3e-2, the output of
    a layer, with up to nine roundings of intermediates on the way to it, 3.8e-3 and 1.9e-2, of two layers in a row 6.2e-3
    and 2.9e-2."""
    rel, most = {"step": (2.8e-3, 1.3e-2), "step_host": (2.8e-3, 1.3e-2), "teacher": (2.1e-3, 1.2e-2),
                 "decoder": (3.8e-3, 1.9e-2), "prefill": (3.8e-3, 1.9e-2), "advance": (6.2e-3, 2.9e-2)}[case["kind"]]
    return {"rel": 4 * rel, "max": 4 * most}


# ---- the same in 64 bits -----------------------------------------------------------------------------------------------


def exact(case, seed):
    """What run() returns, from plain torch in 64 bits, with no rounding between the input and an output."""
    Hq, Hkv, dh, P, C, D, F = _shape(case)
    n, kind = case["n"], case["kind"]
    s = prepare(case, seed)
    torch.cuda.synchronize()
    scale, om = s["scale"], case["out_major"]
    if kind in ("step", "step_host"):
        k, v, seg_k, seg_v = _append(case, s, s["k_new"], s["v_new"])
        out, lse = _attend(s["q"], seg_k, seg_v, s["len0"] + 1, scale, *_prefix(s))
        U = _matmul(out.reshape(n, D), s["w"], om).view(n, P, D)
        if s["bias"] is not None:
            U = U + s["bias"].double().view(P, D)
        oc, _ = _attend(s["q_chunk"], s["kc"], s["vc"], s["clen"], scale)
        lens = s["len0"] + 1
        if kind == "step_host":
            return [[out, lse, oc] if case["lse"] else [out, oc], U, lens, k, v]
        return [out, lse if case["lse"] else None, U, oc, lens, k, v]
    if kind == "teacher":
        return [_causal(s["x"].double(), s["kc"], s["vc"], s["clen"], scale)]
    if kind == "advance":
        a = _matmul(_norm(s["latents"].double(), s["gamma"]), s["w_chunker"], om) + s["b_chunker"].double()
        seen = {}

        def attend(q, k_new, v_new):
            seen["k"], seen["v"], seg_k, seg_v = _append(case, s, k_new, v_new)
            return _attend(q, seg_k, seg_v, s["len0"] + 1, scale)[0]

        x = _layer_exact(a, s["encoder"], s["len0"], case, attend)
        U = _matmul(x, s["w"], om)
        y, kc, vc = _prefill_exact(U.view(n * P, D), s["decoder"], case, s, scale)
        return [a, x, U.view(n, P, D), y.view(n, P, D), s["len0"] + 1, seen["k"], seen["v"], torch.full_like(s["clen"], P), kc, vc]
    if kind == "prefill":
        y, kc, vc = _prefill_exact(s["x"].double().view(n * P, D), s["layer"], case, s, scale)
        return [y.view(n, P, D), torch.full_like(s["clen"], P), kc, vc]
    kc, vc, at = s["kc"].double(), s["vc"].double(), torch.arange(n, device="cuda")

    def attend(q, k_new, v_new):
        kc[at, :, s["clen0"].long()], vc[at, :, s["clen0"].long()] = k_new, v_new
        return _attend(q, kc, vc, s["clen0"] + 1, scale)[0]

    y = _layer_exact(s["x"].double(), s["layer"], s["clen0"], case, attend)
    return [y, s["clen0"] + 1, kc, vc]


def _matmul(x, w, out_major):
    w = w.double()
    return x @ (w.T if out_major else w)


def _norm(x, gamma):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gamma.double()


def _append(case, s, k_new, v_new):
    """The cache with one more row per sequence: as it is stored, and by sequence [n, Hkv, rows, dh]."""
    n, at = case["n"], torch.arange(case["n"], device="cuda")
    k, v, row = s["k"].double(), s["v"].double(), s["len0"].long()
    if not case["paged"]:
        k[at, :, row], v[at, :, row] = k_new.double(), v_new.double()
        return k, v, k, v
    page = s["table"].long()[at, row // PAGE]
    k[page, :, row % PAGE], v[page, :, row % PAGE] = k_new.double(), v_new.double()
    flat = lambda t: t[s["table"].long()].transpose(1, 2).reshape(n, t.shape[1], -1, t.shape[3])
    return k, v, flat(k), flat(v)


def _prefix(s):
    keep = s["kv"]._keep
    return () if keep[3] is None else (keep[3], keep[4])


def _attend(q, k, v, length, scale, k_shared=None, v_shared=None):
    """q [n, Hq, dh] over rows < length of k, v [n, Hkv, rows, dh] and, before them, a prefix of all: (out, log-sum-exp)."""
    n, Hq, dh = q.shape
    Hkv = k.shape[1]
    q, k, v = q.double().reshape(n, Hkv, Hq // Hkv, dh), k.double(), v.double()
    logit = torch.einsum("nhgd,nhsd->nhgs", q, k) * scale
    logit.masked_fill_((torch.arange(k.shape[2], device=q.device) >= length[:, None]).view(n, 1, 1, -1), float("-inf"))
    if k_shared is not None:
        k_shared, v_shared = k_shared[0].double(), v_shared[0].double()
        logit = torch.cat([torch.einsum("nhgd,hsd->nhgs", q, k_shared) * scale, logit], -1)
    lse = torch.logsumexp(logit, -1)
    p = torch.exp(logit - lse[..., None])
    out = torch.einsum("nhgs,nhsd->nhgd", p[..., p.shape[-1] - k.shape[2]:], v)
    if k_shared is not None:
        out = out + torch.einsum("nhgs,hsd->nhgd", p[..., :k_shared.shape[1]], v_shared)
    return out.reshape(n, Hq, dh), lse.reshape(n, Hq)


def _causal(q, k, v, length, scale):
    """q [n, rows, Hq, dh]: position t sees rows 0..t; a position that does not exist is zero."""
    out = torch.empty_like(q)
    for t in range(q.shape[1]):
        out[:, t] = _attend(q[:, t], k[:, :, :t + 1], v[:, :, :t + 1], torch.full_like(length, t + 1), scale)[0]
    return out * (torch.arange(q.shape[1], device=q.device) < length[:, None])[:, :, None, None]


def _layer_exact(x, layer, pos, case, attend):
    Hq, Hkv, dh, _, _, D, F = _shape(case)
    g1, wqkv, wo, g2, wgu, wdown = layer._keep
    om, rows = case["out_major"], x.shape[0]
    qkv = _matmul(_norm(x, g1), wqkv, om).view(rows, Hq + 2 * Hkv, dh)
    angle = pos.double()[:, None] * 10000.0 ** (-torch.arange(dh // 2, device="cuda", dtype=torch.float64) * 2 / dh)
    c, sn = angle.cos()[:, None], angle.sin()[:, None]
    a, b = qkv[:, :Hq + Hkv, :dh // 2], qkv[:, :Hq + Hkv, dh // 2:]
    qk = torch.cat([a * c - b * sn, b * c + a * sn], -1)
    h = x + _matmul(attend(qk[:, :Hq], qk[:, Hq:], qkv[:, Hq + Hkv:]).reshape(rows, D), wo, om)
    gu = _matmul(_norm(h, g2), wgu, om)
    return h + _matmul(torch.nn.functional.silu(gu[:, :F]) * gu[:, F:], wdown, om)


def _prefill_exact(x, layer, case, s, scale):
    Hq, Hkv, dh, P, _, _, _ = _shape(case)
    n = case["n"]
    kc, vc = s["kc"].double(), s["vc"].double()

    def attend(q, k_new, v_new):
        kc[:, :, :P], vc[:, :, :P] = (t.view(n, P, Hkv, dh).transpose(1, 2) for t in (k_new, v_new))
        full = torch.full((n,), P, dtype=torch.int32, device="cuda")
        return _causal(q.reshape(n, P, Hq, dh), kc[:, :, :P], vc[:, :, :P], full, scale)

    return _layer_exact(x, layer, torch.arange(P, device="cuda").repeat(n), case, attend), kc, vc
