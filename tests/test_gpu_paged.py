"""A paged coarse cache gives the results of the contiguous cache it stands for:
append bit-exactly, attention within the usual bar of the CPU oracle (which sees the
contiguous cache; a paged cache is a storage layout, not another computation)."""
import numpy as np
import pytest
import torch

import paper_2512_20687_b200 as ph
from paper_2512_20687_b200 import workloads as wl

from gpu_util import Ctx, assert_close, dev_bf16, dev_i32, host_bits, host_f64

pytestmark = pytest.mark.gpu

NT = 16


def cfg_small(i, **kw):
    return wl.scaled(wl.CONFIGS[i], **kw)


def to_pages(a, table, page_rows, n_pages, fill):
    """Contiguous [n_units, Hkv, cap, dh] -> pool [n_pages, Hkv, page_rows, dh] through the table."""
    n_units, Hkv, cap, dh = a.shape
    pool = np.full((n_pages, Hkv, page_rows, dh), fill, np.uint16)
    for u in range(n_units):
        for j in range(table.shape[1]):
            pool[table[u, j]] = a[u, :, j * page_rows:(j + 1) * page_rows]
    return pool


def from_pages(pool, table, page_rows):
    n_units, ppu = table.shape
    return np.concatenate([pool[table[:, j]] for j in range(ppu)], axis=2)


@pytest.mark.parametrize("idx,B,S,page_rows", [(1, 9, 701, 64), (1, 64, 512, 128), (4, 40, 128, 64), (0, 2, 16, 64)])
def test_paged_append_and_attention(oracle, idx, B, S, page_rows):
    cfg = cfg_small(idx, B=B, S=S)
    co = wl.coarse_inputs(cfg, poison=True)
    ppu = -(-S // page_rows)
    cap = ppu * page_rows
    lens = np.array([max(0, S - 1 - 37 * (u % 5)) for u in range(B)], np.int32)
    lens[0] = S - 1
    if B > 2:
        lens[1], lens[2] = 0, page_rows - 1                      # an empty unit; an append that fills a page
    pad = lambda a: np.concatenate([a, np.full(a.shape[:2] + (cap - S, a.shape[3]), 0x7FC1, np.uint16)], axis=2)
    k, v = pad(co["k"]), pad(co["v"])
    for u, n in enumerate(lens):
        k[u, :, n:] = 0x7FC1
        v[u, :, n:] = 0xFFC1
    n_pages = B * ppu + 3
    table = np.random.default_rng(idx).permutation(n_pages)[: B * ppu].reshape(B, ppu).astype(np.int32)
    scale = cfg.dh ** -0.5
    ok, ov, ol = k.copy(), v.copy(), lens.copy()
    assert oracle.kv_append(ok, ov, ol, co["k_new"], co["v_new"]) == 0
    want, want_lse = oracle.attention(co["q"], ok, ov, ol, scale, n_threads=NT)
    with Ctx(cfg) as c:
        pk, pv = dev_bf16(to_pages(k, table, page_rows, n_pages, 0x7FC1)), dev_bf16(to_pages(v, table, page_rows, n_pages, 0x7FC1))
        dl = dev_i32(lens)
        kv = ph.make_kv(pk, pv, dl, page_table=dev_i32(table))
        assert kv.cap == cap and kv.n_units == B
        ph.photon_kv_append(c.h, kv, dev_bf16(co["k_new"]), dev_bf16(co["v_new"]))
        q = dev_bf16(co["q"])
        out = torch.empty_like(q)
        lse = torch.empty(B, cfg.Hq, dtype=torch.float32, device="cuda")
        ph.photon_coarse_attn(c.h, kv, q, out, lse, scale)
        out2 = torch.empty_like(q)
        ph.photon_flat_attn(c.h, kv, q, out2, None, scale)
        assert c.status() == 0
        assert np.array_equal(dl.cpu().numpy(), ol)
        gk, gv = from_pages(host_bits(pk), table, page_rows), from_pages(host_bits(pv), table, page_rows)
        assert np.array_equal(gk, ok) and np.array_equal(gv, ov)         # the append wrote the right page, bit-exactly
    assert_close(host_f64(out), want, "paged coarse attention")
    assert np.array_equal(host_bits(out), host_bits(out2))
    fin = np.isfinite(want_lse)
    assert np.abs(lse.cpu().numpy()[fin] - want_lse[fin]).max() < 2e-3


def test_paged_and_contiguous_give_the_same_bits():
    cfg = cfg_small(1, B=16, S=8192)
    co = wl.coarse_inputs(cfg)
    page_rows, ppu = 256, 32
    n_pages = cfg.B * ppu
    table = np.random.default_rng(7).permutation(n_pages).reshape(cfg.B, ppu).astype(np.int32)
    scale = cfg.dh ** -0.5
    with Ctx(cfg) as c:
        q = dev_bf16(co["q"])
        a, b = torch.empty_like(q), torch.empty_like(q)
        dl = dev_i32(co["len"])
        ph.photon_coarse_attn(c.h, ph.make_kv(dev_bf16(co["k"]), dev_bf16(co["v"]), dl), q, a, None, scale)
        pk, pv = dev_bf16(to_pages(co["k"], table, page_rows, n_pages, 0)), dev_bf16(to_pages(co["v"], table, page_rows, n_pages, 0))
        ph.photon_coarse_attn(c.h, ph.make_kv(pk, pv, dl, page_table=dev_i32(table)), q, b, None, scale)
        assert c.status() == 0
    assert np.array_equal(host_bits(a), host_bits(b))                    # the same tiles in the same order


def test_bad_pages_and_calls_that_do_not_take_pages():
    cfg = cfg_small(0, B=2, S=16)
    co = wl.coarse_inputs(cfg)
    pool = np.zeros((3, cfg.Hkv, 64, cfg.dh), np.uint16)
    with Ctx(cfg) as c:
        pk, pv, dl = dev_bf16(pool), dev_bf16(pool), dev_i32(co["len"])
        kv = ph.make_kv(pk, pv, dl, page_table=dev_i32(np.array([[1], [5]], np.int32)))
        ph.photon_kv_append(c.h, kv, dev_bf16(co["k_new"]), dev_bf16(co["v_new"]))
        assert c.status() == ph.PHOTON_DEV_BAD_INDEX                      # unit 1 names page 5 of 3
        assert list(dl.cpu().numpy()) == [co["len"][0] + 1, co["len"][1]]
        q = dev_bf16(co["q"])
        out = torch.empty_like(q)
        ph.photon_coarse_attn(c.h, kv, q, out, None, 1.0)
        assert c.status() == ph.PHOTON_DEV_BAD_INDEX and np.isfinite(host_f64(out)).all()
        q1, o1 = q.unsqueeze(1).contiguous(), out.unsqueeze(1).contiguous()
        for call in (lambda: ph.photon_chunk_attn(c.h, kv, q, None, out),
                     lambda: ph.photon_chunk_causal_attn(c.h, kv, q1, None, o1)):
            with pytest.raises(ph.PhotonError) as e:
                call()
            assert e.value.code == ph.PHOTON_ERR_INVALID_ARG
        kv.page_rows = 48                                                 # not a multiple of 64
        with pytest.raises(ph.PhotonError):
            ph.photon_coarse_attn(c.h, kv, q, out, None, 1.0)


@pytest.mark.parametrize("Hq,Hkv,dh", [(16, 4, 128), (8, 8, 128), (4, 2, 64)])
def test_step_on_pages_appends_inside_the_attention(Hq, Hkv, dh):
    """The step folds the append into the attention for paged caches too: against append and attention called one after the
    other, same bits, same cache, lengths and status.  Units that are empty, one row short of a page, at a page's first row,
    full, and one whose next page does not exist."""
    cfg = wl.scaled(wl.CONFIGS[1], B=9, Hq=Hq, Hkv=Hkv, dh=dh, D=Hq * dh)
    B, page_rows, ppu, P = 9, 128, 3, cfg.P
    n_pages, cap, scale = B * ppu, 384, dh ** -0.5
    g = torch.Generator("cuda").manual_seed(Hq)

    def rand(*shape, std=1.0):
        return (torch.randn(*shape, generator=g, device="cuda") * std).to(torch.bfloat16)

    lens = np.array([0, 63, 64, 127, 128, 200, cap, 255, 256], np.int32)
    table = np.random.default_rng(3).permutation(n_pages).reshape(B, ppu).astype(np.int32)
    table[8, 2] = n_pages                                                # unit 8 is at the first row of a page that is not there
    table_dev, pk, pv = dev_i32(table), rand(n_pages, Hkv, page_rows, dh), rand(n_pages, Hkv, page_rows, dh)
    k_new, v_new, q, w = rand(B, Hkv, dh), rand(B, Hkv, dh), rand(B, Hq, dh), rand(Hq * dh, P * Hq * dh, std=0.02)
    got = []
    with Ctx(cfg) as c:
        for folded in (False, True):
            k, v, ln = pk.clone(), pv.clone(), dev_i32(lens)
            kv = ph.make_kv(k, v, ln, page_table=table_dev)
            out, lse = torch.empty_like(q), torch.empty(B, Hq, device="cuda")
            n0 = ph.photon_launch_count(c.h)
            if folded:
                U = torch.empty(B, P, Hq * dh, dtype=torch.bfloat16, device="cuda")
                args = ph.make_step_args(kv, k_new, v_new, q, out, scale, w, ph.PHOTON_W_IN_MAJOR, U, B, lse_coarse=lse)
                ph.photon_decode_step(c.h, args)
                assert ph.photon_launch_count(c.h) - n0 == 2
            else:
                ph.photon_kv_append(c.h, kv, k_new, v_new)
                ph.photon_coarse_attn(c.h, kv, q, out, lse, scale)
            assert c.status() == ph.PHOTON_DEV_CAPACITY | ph.PHOTON_DEV_BAD_INDEX
            got.append([host_bits(t) for t in (out, k, v)] + [lse.cpu().numpy(), ln.cpu().numpy()])
    assert np.array_equal(got[0][-1], lens + np.array([1, 1, 1, 1, 1, 1, 0, 1, 0]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n,S,lengths", [(80, 1100, "ragged"), (80, 1024, "equal"), (75, 1088, "equal"), (3, 3000, "ragged"), (300, 70, "ragged"),
                                         (20, 1300, "one long"), (70, 2200, "ragged")])
@pytest.mark.parametrize("paged", [False, True])
def test_streams_at_the_edges_of_the_deal(n, S, lengths, paged):
    """More streams than CTAs, lengths equal (fewer CTAs take part) and not, streams of 16 tiles and of 17, of 64 features (cut above 8).  Within the two roundings to bf16 of torch in 64 bits: the output's (2^-8 of the value) and the weights' (2^-8
    of the weighted sum of the absolute values)."""
    Hq, Hkv, dh = 8, 4, 64
    cfg = wl.scaled(wl.CONFIGS[1], B=n, Hq=Hq, Hkv=Hkv, dh=dh, D=Hq * dh)
    rng = np.random.default_rng(n)
    lens = (np.full(n, S) if lengths == "equal" else rng.integers(0, S + 1, n) if lengths == "ragged" else np.where(np.arange(n) == 7, S, 40)).astype(np.int32)
    g = torch.Generator("cuda").manual_seed(n)
    k, v, q = ((torch.randn(*s, generator=g, device="cuda")).to(torch.bfloat16) for s in ((n, Hkv, S, dh), (n, Hkv, S, dh), (n, Hq, dh)))
    out, lse = torch.empty_like(q), torch.empty(n, Hq, device="cuda")
    with Ctx(cfg) as c:
        if paged:
            ppu = -(-S // 64)
            pad = lambda t: torch.nn.functional.pad(t, (0, 0, 0, ppu * 64 - S)).view(n, Hkv, ppu, 64, dh).transpose(1, 2).reshape(n * ppu, Hkv, 64, dh)
            order = torch.randperm(n * ppu, generator=g, device="cuda")
            pk, pv = torch.empty_like(pad(k)), torch.empty_like(pad(v))
            pk[order], pv[order] = pad(k), pad(v)
            kv = ph.make_kv(pk, pv, dev_i32(lens), page_table=order.to(torch.int32).view(n, ppu).contiguous())
        else:
            kv = ph.make_kv(k, v, dev_i32(lens))
        ph.photon_coarse_attn(c.h, kv, q, out, lse, dh ** -0.5)
        assert c.status() == 0
    logit = torch.einsum("nhgd,nhsd->nhgs", q.double().view(n, Hkv, Hq // Hkv, dh), k.double()) * dh ** -0.5
    logit.masked_fill_((torch.arange(S, device="cuda") >= torch.from_numpy(lens).cuda()[:, None])[:, None, None], float("-inf"))
    w = torch.softmax(logit, -1).nan_to_num(0.0)
    want, size = (torch.einsum("nhgs,nhsd->nhgd", w, x).reshape(n, Hq, dh) for x in (v.double(), v.double().abs()))
    assert ((out.double() - want).abs() <= 2.0 ** -8 * (want.abs() + size) + 1e-5).all()
    want_lse = torch.logsumexp(logit, -1).view(n, Hq)
    fin = torch.isfinite(want_lse)
    assert torch.equal(torch.isneginf(lse), ~fin) and (lse.double() - want_lse)[fin].abs().max() < 2e-3


# tile counts of the units before the append and after it: equal and all open a tile (one, two, eighteen tiles: streams that are cut);
# equal and none does; equal only before; equal only after
BEHIND_AN_APPEND = [(64,), (128,), (1088,), (127,), (0,), (63, 64), (1087, 1088), (64, 65), (1089, 1088)]


@pytest.mark.parametrize("lengths", BEHIND_AN_APPEND)
@pytest.mark.parametrize("n", [77, 80])
@pytest.mark.parametrize("paged", [False, True])
def test_deal_of_more_streams_than_ctas_behind_an_append(n, lengths, paged):
    """More streams than CTAs: how many CTAs take part depends on whether the tile counts are equal, and the attention deals while
    the append in front of it writes the lengths.  Behind reads of varied length (the probe), so that its CTAs meet the append at
    different points: the bits of a call on an idle device each time, also of a second attention (tickets and counters are
    as they should be), status clear, and the result within its two roundings to bf16 of torch in 64 bits: the output's (2^-8 of the
    value) and the weights' (2^-8 of the weighted sum of the absolute values)."""
    Hq, Hkv, dh, S = 8, 4, 64, 64 * (max(lengths) // 64 + 1)
    cfg = wl.scaled(wl.CONFIGS[1], B=n, Hq=Hq, Hkv=Hkv, dh=dh, D=Hq * dh)
    g = torch.Generator("cuda").manual_seed(n + len(lengths) + S)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    len0 = dev_i32([lengths[u % len(lengths)] for u in range(n)])
    k, v, q, k_new, v_new = rand(n, Hkv, S, dh), rand(n, Hkv, S, dh), rand(n, Hq, dh), rand(n, Hkv, dh), rand(n, Hkv, dh)
    ln, ppu = len0.clone(), S // 64
    at = torch.arange(n, device="cuda")
    want_k, want_v = k.double(), v.double()
    want_k[at, :, len0.long()], want_v[at, :, len0.long()] = k_new.double(), v_new.double()
    if paged:
        order = torch.randperm(n * ppu, generator=g, device="cuda")
        cut = lambda t: t.view(n, Hkv, ppu, 64, dh).transpose(1, 2).reshape(n * ppu, Hkv, 64, dh)
        pk, pv = torch.empty_like(cut(k)), torch.empty_like(cut(v))
        pk[order], pv[order] = cut(k), cut(v)
        kv = ph.make_kv(pk, pv, ln, page_table=order.to(torch.int32).view(n, ppu).contiguous())
    else:
        kv = ph.make_kv(k, v, ln)
    held = torch.empty(64 << 20, dtype=torch.uint8, device="cuda").random_()
    scale, first = dh ** -0.5, None
    with Ctx(cfg) as c:
        for turn in range(60):
            outs = [(torch.empty_like(q), torch.empty(n, Hq, device="cuda")) for _ in range(2)]
            ln.copy_(len0)
            torch.cuda.synchronize()
            if turn:
                ph.photon_read_probe(c.h, held[:(turn * 1237 % 4096) * 16384])      # 0 to 64 MB
            ph.photon_kv_append(c.h, kv, k_new, v_new)
            if not turn:
                torch.cuda.synchronize()
            for out, lse in outs:
                ph.photon_coarse_attn(c.h, kv, q, out, lse, scale)
            assert c.status() == 0
            got = [torch.cat([out.view(torch.int16).int().view(n, -1), lse.view(torch.int32)], 1) for out, lse in outs]
            first = got[0] if first is None else first
            assert torch.equal(got[0], first) and torch.equal(got[1], first), turn
            assert torch.equal(ln, len0 + 1)
    out, lse = outs[0]
    logit = torch.einsum("nhgd,nhsd->nhgs", q.double().view(n, Hkv, Hq // Hkv, dh), want_k) * scale
    logit.masked_fill_((torch.arange(S, device="cuda") > len0[:, None])[:, None, None], float("-inf"))
    w = torch.softmax(logit, -1)
    want, size = (torch.einsum("nhgs,nhsd->nhgd", w, x).reshape(n, Hq, dh) for x in (want_v, want_v.abs()))
    assert ((out.double() - want).abs() <= 2.0 ** -8 * (want.abs() + size) + 1e-5).all()
    assert (lse.double() - torch.logsumexp(logit, -1).view(n, Hq)).abs().max() < 2e-3


# (16, 4): kept whole, cut in halves, cut in four; ragged with all CTAs, few tiles per CTA, many; nearly equal.  (16, 1): cut in two and four,
# ragged, nearly equal.  (8, 8): never whole above 8 tiles
DEALS = [(16, 4, 32, 640, "equal"), (16, 4, 32, 1024, "equal"), (16, 4, 24, 1024, "equal"), (16, 4, 16, 1024, "equal"), (16, 4, 75, 576, "equal"),
         (16, 4, 75, 1000, "ragged"), (16, 4, 250, 300, "ragged"), (16, 4, 60, 3000, "ragged"), (16, 4, 32, 1000, "ragged"), (16, 4, 75, 800, "near"),
         (16, 1, 100, 1024, "equal"), (16, 1, 64, 1024, "equal"), (16, 1, 300, 1000, "ragged"), (16, 1, 130, 900, "near"), (8, 8, 37, 1024, "equal"),
         (8, 8, 37, 1000, "ragged")]


@pytest.mark.parametrize("Hq,Hkv,n,S,lengths", DEALS)
def test_streams_that_stay_whole_and_streams_that_are_cut(Hq, Hkv, n, S, lengths):
    """Heads of 128 features, where what a cut costs decides.  Twice (the tickets are as they should be), and within the two
    roundings to bf16 of torch in 64 bits: the output's (2^-8 of the value) and the weights' (2^-8 of the weighted sum of the absolute values)."""
    dh = 128
    cfg = wl.scaled(wl.CONFIGS[1], B=n, Hq=Hq, Hkv=Hkv, dh=dh, D=Hq * dh)
    rng = np.random.default_rng(n + S)
    lens = dev_i32(np.full(n, S) if lengths == "equal" else rng.integers(0 if lengths == "ragged" else S * 7 // 8, S + 1, n))
    g = torch.Generator("cuda").manual_seed(n)
    k, v, q = ((torch.randn(*s, generator=g, device="cuda")).to(torch.bfloat16) for s in ((n, Hkv, S, dh), (n, Hkv, S, dh), (n, Hq, dh)))
    outs = [(torch.empty_like(q), torch.empty(n, Hq, device="cuda")) for _ in range(2)]
    with Ctx(cfg) as c:
        for out, lse in outs:
            ph.photon_coarse_attn(c.h, ph.make_kv(k, v, lens), q, out, lse, dh ** -0.5)
            assert c.status() == 0
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16)) and torch.equal(outs[0][1], outs[1][1])
    out, lse = outs[0]
    for u in range(n):                                                    # (a unit at a time: 64-bit copies of the caches are large)
        L = int(lens[u])
        if L == 0:
            assert bool((out[u] == 0).all()) and bool(torch.isneginf(lse[u]).all())
            continue
        logit = torch.einsum("hgd,hsd->hgs", q[u].double().view(Hkv, Hq // Hkv, dh), k[u, :, :L].double()) * dh ** -0.5
        w = torch.softmax(logit, -1)
        want, size = (torch.einsum("hgs,hsd->hgd", w, x).reshape(Hq, dh) for x in (v[u, :, :L].double(), v[u, :, :L].double().abs()))
        assert ((out[u].double() - want).abs() <= 2.0 ** -8 * (want.abs() + size) + 1e-5).all(), u
        assert (lse[u].double() - torch.logsumexp(logit, -1).view(Hq)).abs().max() < 2e-3
