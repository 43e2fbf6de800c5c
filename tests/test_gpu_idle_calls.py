"""The public entry points called the way a host loop without graphs calls them: one call at a
time, each on an idle device, many times over.  Kernels that overlap their predecessor's tail
(programmatic dependent launch) start under other conditions here than inside a replayed graph
or a tight sequence of launches, and a fault that shows once in some tens of such calls does not
show in a parity test that calls once.  Every call must leave the status word clear and, where
the inputs are put back, give the first call's bits."""
import numpy as np
import pytest
import torch

import paper_2512_20687_b200 as ph
from paper_2512_20687_b200 import workloads as wl

from gpu_util import Ctx, chunks_to_dev, coarse_to_dev, dev_bf16

pytestmark = pytest.mark.gpu

CALLS = 120


def bits(t):
    return t.view(torch.int16)


def test_layer_steps_one_at_a_time_on_the_default_workload():
    """STEP of an encoder layer on the coarse caches and of a decoder layer on the chunk buffers
    (64 and 128 rows: the shapes of the default workload), the lengths put back before every call."""
    cfg = wl.CONFIGS[1]
    s = wl.step_inputs(cfg)
    co, chk = s["coarse"], s["chunks"]
    scale = cfg.dh ** -0.5
    li = wl.encoder_layer_inputs(cfg)
    names = ("g1", "wqkv", "wo", "g2", "wgu", "wdown")
    with Ctx(cfg) as c:
        d, dc = coarse_to_dev(co), chunks_to_dev(chk)
        layer = ph.make_layer(*(dev_bf16(li[n]) for n in names), ph.PHOTON_W_IN_MAJOR, li["F"])
        scr = ph.make_layer_scratch(max(cfg.B, cfg.Nc), cfg.Hq, cfg.Hkv, cfg.dh, li["F"], torch.device("cuda"),
                                    torch.bfloat16)
        ex = dev_bf16(li["x"])
        ey, ey0 = torch.empty_like(ex), None
        len0 = d["len"].clone()
        for it in range(CALLS):
            d["len"].copy_(len0)
            torch.cuda.synchronize()
            ph.photon_encoder_step(c.h, layer, scr, ex, d["kv"], ey, scale=scale)
            torch.cuda.synchronize()
            assert c.status() == 0, f"encoder step, call {it}"
            if ey0 is None:
                ey0 = ey.clone()
            assert torch.equal(bits(ey), bits(ey0)), f"encoder step, call {it}"
        gen = torch.Generator(device="cuda")
        gen.manual_seed(5)
        dx = torch.empty(cfg.Nc, cfg.D, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
        dy, dy0 = torch.empty_like(dx), None
        clen0 = (dc["len"] - 1).clamp(min=0)
        for it in range(CALLS):
            dc["len"].copy_(clen0)
            torch.cuda.synchronize()
            ph.photon_decoder_step(c.h, layer, scr, dx, dc["kv"], dy, scale=scale)
            torch.cuda.synchronize()
            assert c.status() == 0, f"decoder step, call {it}"
            if dy0 is None:
                dy0 = dy.clone()
            assert torch.equal(bits(dy), bits(dy0)), f"decoder step, call {it}"


@pytest.mark.parametrize("idx", [1, 3])
def test_decode_steps_one_at_a_time(idx):
    """The four-part decode step (append folded in or not, a shared prefix with the own keys riding along on
    workload 3), the lengths put back before every call."""
    cfg = wl.CONFIGS[idx]
    s = wl.step_inputs(cfg)
    co, cv, chk = s["coarse"], s["converter"], s["chunks"]
    scale = cfg.dh ** -0.5
    with Ctx(cfg) as c:
        d, dc = coarse_to_dev(co), chunks_to_dev(chk)
        len0 = d["len"].clone()
        out = torch.empty_like(d["q"])
        U = torch.empty(cfg.B, cfg.P, cfg.D, dtype=torch.bfloat16, device="cuda")
        oc = torch.empty_like(dc["q"])
        args = ph.make_step_args(d["kv"], d["k_new"], d["v_new"], d["q"], out, scale, dev_bf16(cv["w_in_major"]),
                                 ph.PHOTON_W_IN_MAJOR, U, cfg.B, chunks=dc["kv"], q_chunk=dc["q"], out_chunk=oc,
                                 Nc=cfg.Nc, scale_chunk=scale)
        first = None
        for it in range(CALLS):
            d["len"].copy_(len0)
            torch.cuda.synchronize()
            ph.photon_decode_step(c.h, args)
            torch.cuda.synchronize()
            assert c.status() == 0, f"decode step, call {it}"
            if first is None:
                first = (out.clone(), U.clone(), oc.clone())
            for got, want in zip((out, U, oc), first):
                assert torch.equal(bits(got), bits(want)), f"decode step, call {it}"
        assert np.array_equal(d["len"].cpu().numpy(), len0.cpu().numpy() + 1)


@pytest.mark.parametrize("B", [0, 3])
def test_small_steps_without_a_coarse_sequence_behind_writers_of_their_chunks(B):
    """No coarse sequence is there, so no kernel of the step waits before the chunk attention but the converter (B latents), which
    lets the next kernel start at once; the queries, the chunks' new rows and their lengths come from kernels of the library
    enqueued just before.  Against the same calls with a wait between them."""
    Hq, Hkv, dh, P, C, Nc = 4, 2, 64, 4, 8, 24
    D = Hq * dh
    cfg = wl.scaled(wl.CONFIGS[0], B=1, Hq=Hq, Hkv=Hkv, dh=dh, D=D, P=P, C=C)
    gen = torch.Generator("cuda").manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    k0, v0, xs, wq = rand(Nc, Hkv, P + C, dh), rand(Nc, Hkv, P + C, dh), rand(C, Nc, D), rand(D, D)
    k_new, v_new = rand(C, Nc, Hkv, dh), rand(C, Nc, Hkv, dh)
    x, w, one = rand(max(B, 1), D), rand(D, P * D), torch.zeros(1, 1, 1, dh, dtype=torch.bfloat16, device="cuda")
    held = torch.empty(16 << 20, dtype=torch.uint8, device="cuda").random_()
    with Ctx(cfg, max_queries=Nc) as c:
        first = None
        for turn in range(20):
            kc, vc, ln = k0.clone(), v0.clone(), torch.full((Nc,), P, dtype=torch.int32, device="cuda")
            ckv, none = ph.make_kv(kc, vc, ln), ph.make_kv(one, one.clone(), torch.zeros(1, dtype=torch.int32, device="cuda"))
            none.n_units = 0
            q, outs, U = torch.empty(Nc, D, dtype=torch.bfloat16, device="cuda"), [], torch.empty(max(B, 1), P, D, dtype=torch.bfloat16, device="cuda")
            torch.cuda.synchronize()
            if turn:
                ph.photon_read_probe(c.h, held[:turn * 839680])
            for t in range(C):
                outs.append(torch.empty(Nc, Hq, dh, dtype=torch.bfloat16, device="cuda"))
                args = ph.make_step_args(none, one, one, one, one, 1.0, w, ph.PHOTON_W_IN_MAJOR, U, B, chunks=ckv, q_chunk=q.view(Nc, Hq, dh),
                                         out_chunk=outs[-1], Nc=Nc, scale_chunk=dh ** -0.5, x=x)
                ph.photon_linear(c.h, xs[t], wq, ph.PHOTON_W_IN_MAJOR, None, q)
                ph.photon_kv_append(c.h, ckv, k_new[t], v_new[t])
                if not turn:
                    torch.cuda.synchronize()
                ph.photon_decode_step(c.h, args)
                if not turn:
                    torch.cuda.synchronize()
            assert c.status() == 0
            got = [bits(o).clone() for o in outs] + [bits(U).clone() if B else None]
            first = first or got
            for a, b in zip(got, first):
                assert a is None or torch.equal(a, b), turn


@pytest.mark.parametrize("Hq,Hkv,dh,P,C,B,S,per", [(16, 4, 128, 4, 4, 20, 300, 2), (16, 4, 128, 8, 16, 20, 300, 2), (16, 4, 128, 4, 12, 9, 100, 3), (8, 8, 128, 8, 16, 12, 200, 2),
                                                   (8, 8, 128, 8, 16, 40, 200, 2), (8, 4, 128, 8, 16, 20, 200, 2), (8, 4, 128, 8, 16, 20, 40, 2),
                                                   (4, 2, 64, 4, 4, 5, 20, 4)])
def test_captured_steps_in_either_order_of_their_attentions(Hq, Hkv, dh, P, C, B, S, per):
    """A captured step enqueues the chunk attention in front of the coarse attention or behind it; replayed, the bits of the same step
    called by itself."""
    cfg = wl.scaled(wl.CONFIGS[1], B=B, Hq=Hq, Hkv=Hkv, dh=dh, D=Hq * dh, P=P, C=C)
    D, Nc = Hq * dh, B * per
    gen = torch.Generator("cuda").manual_seed(B + S)
    rand = lambda *s, std=1.0: (torch.randn(*s, generator=gen, device="cuda") * std).to(torch.bfloat16)
    k, v, q, k_new, v_new = rand(B, Hkv, S, dh), rand(B, Hkv, S, dh), rand(B, Hq, dh), rand(B, Hkv, dh), rand(B, Hkv, dh)
    kc, vc, qc, w = rand(Nc, Hkv, P + C, dh), rand(Nc, Hkv, P + C, dh), rand(Nc, Hq, dh), rand(D, P * D, std=D ** -0.5)
    len0 = torch.randint(0, S, (B,), generator=gen, device="cuda", dtype=torch.int32)
    ln, lc = len0.clone(), torch.randint(P, P + C + 1, (Nc,), generator=gen, device="cuda", dtype=torch.int32)
    out, oc, U = torch.empty_like(q), torch.empty_like(qc), torch.empty(B, P, D, dtype=torch.bfloat16, device="cuda")
    with Ctx(cfg, max_queries=Nc) as c:
        args = ph.make_step_args(ph.make_kv(k, v, ln), k_new, v_new, q, out, dh ** -0.5, w, ph.PHOTON_W_IN_MAJOR, U, B, chunks=ph.make_kv(kc, vc, lc),
                                 q_chunk=qc, out_chunk=oc, Nc=Nc, scale_chunk=dh ** -0.5)
        ph.photon_decode_step(c.h, args)
        want = [bits(t).clone() for t in (out, U, oc)]
        stream = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            ln.copy_(len0)
            ph.photon_decode_step(c.h, args, stream=stream)
        for _ in range(5):
            for t in (out, U, oc):
                t.fill_(7.0)
            graph.replay()
            torch.cuda.synchronize()
            assert c.status() == 0 and torch.equal(ln, len0 + 1)
            for got, b in zip((out, U, oc), want):
                assert torch.equal(bits(got), b)
        del graph
