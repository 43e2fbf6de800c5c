"""Parity of the context chunker's two kernels (row normalisation, linear map on
the tensor cores incl. its split of K over a cluster) with the CPU oracle, through
the C boundary.  bf16 outputs: max abs error 2e-2, mean abs error 2e-3 against the
fp64 oracle on the same bf16 inputs."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2512_20687_b200 as ph
from paper_2512_20687_b200 import workloads as wl

from gpu_util import Ctx, assert_close, dev_bf16, host_bits, host_f64

pytestmark = pytest.mark.gpu

NT = 16     # oracle threads


def cfg_small(i, **kw):
    return wl.scaled(wl.CONFIGS[i], **kw)


@pytest.mark.parametrize("rows,cols,with_gamma", [(64, 8192, True), (5, 4096, False), (3, 8, True), (130, 1032, True),
                                                  (3000, 1032, True), (1025, 2048, False), (1500, 8, True)])
def test_rmsnorm_matches_oracle(oracle, rows, cols, with_gamma):
    x = wl.normal_bf16(21, "x", (rows, cols), std=3.0)
    g = wl.f32_to_bf16_bits((wl.bf16_bits_to_f64(wl.normal_bf16(21, "g", (cols,), std=0.2)) + 1.0).astype(np.float32))
    want = oracle.rmsnorm(x, g if with_gamma else None, eps=1e-5)
    with Ctx(cfg_small(0)) as c:
        dx = dev_bf16(x)
        out = torch.full_like(dx, 9.0)
        ph.photon_rmsnorm(c.h, dx, dev_bf16(g) if with_gamma else None, 1e-5, out)
        assert c.status() == 0
        inplace = dx.clone()
        ph.photon_rmsnorm(c.h, inplace, dev_bf16(g) if with_gamma else None, 1e-5, inplace)
        assert c.status() == 0
    assert_close(host_f64(out), want, f"rmsnorm {rows}x{cols}")
    assert np.array_equal(host_bits(out), host_bits(inplace))
    # bf16 rounding of an O(1) value: within one bf16 step of the oracle's own rounding
    assert np.abs(host_f64(out) - wl.bf16_bits_to_f64(oracle.round_bf16(want))).max() <= 2.0 ** -6


# (B, K, N): the 1B-class chunker (4 CTAs share a tile), the chunk-parallel one (wide batch),
# a tile count that needs no split, odd batch sizes, the smallest K that is still split, K too short to split
# and more narrow tiles than SMs (wider slabs, one wave)
SHAPES = [(64, 8192, 2048), (512, 4096, 1024), (64, 2048, 8192), (1, 1024, 64), (130, 1024, 128),
          (17, 512, 64), (200, 4096, 256), (64, 1024, 11264), (130, 512, 6400),
          # thousands of rows: the persistent kernel (one to several tiles per CTA, a ragged last row tile)
          (9000, 512, 1280), (16384, 256, 768), (4100, 192, 2816)]


@pytest.mark.parametrize("B,K,N", SHAPES)
@pytest.mark.parametrize("out_major", [False, True])
def test_linear_matches_oracle(oracle, B, K, N, out_major):
    x = wl.normal_bf16(22, "x", (B, K))
    w = wl.normal_bf16(22, "w", (K, N), std=K ** -0.5)
    bias = wl.normal_bf16(22, "b", (N,), std=0.5)
    wm = np.ascontiguousarray(w.T) if out_major else w
    want = oracle.linear(x, wm, bias, w_out_major=out_major, n_threads=NT)
    with Ctx(cfg_small(0)) as c:
        y = torch.full((B, N), 7.0, dtype=torch.bfloat16, device="cuda")
        layout = ph.PHOTON_W_OUT_MAJOR if out_major else ph.PHOTON_W_IN_MAJOR
        ph.photon_linear(c.h, dev_bf16(x), dev_bf16(wm), layout, dev_bf16(bias), y)
        y2 = torch.empty_like(y)
        ph.photon_linear(c.h, dev_bf16(x), dev_bf16(wm), layout, dev_bf16(bias), y2)
        assert c.status() == 0
    assert np.array_equal(host_bits(y), host_bits(y2))                  # the split of K adds in a fixed order
    assert_close(host_f64(y), want, f"linear {B}x{K}x{N}")


def cut_of(c, B, K, N, gated=False):
    """(columns per tile, CTAs per tile, ring stages, MMA warps) that the library takes on this device."""
    clusters, out = (ctypes.c_int32 * 9)(), (ctypes.c_int32 * 4)()
    ph.load().photon_internal_clusters(c.h, clusters)
    ph.load().photon_internal_projection_cut(clusters, B, K, N, int(gated), out)
    return tuple(out)


@pytest.mark.parametrize("N", [11264, 9536])
def test_linear_with_more_tiles_than_sms_repeated_on_an_idle_device(N):
    """128 rows and 88 tiles of 128 output columns (the gate/up projection of a layer step on 128 chunks), or 149 of 64, more than
    SMs: 200 calls, each on an idle device with another kernel run in between, as a caller that launches one operation at a
    time does.  Every call gives the first call's bits and leaves the status word clear.  (A form of this kernel that put
    two CTAs on an SM for such tile counts gave up on a wait, or failed, once in some tens of such calls.)"""
    B, K = 128, 2048
    x = dev_bf16(wl.normal_bf16(25, "x", (B, K)))
    w = dev_bf16(wl.normal_bf16(25, "w", (K, N), std=K ** -0.5))
    with Ctx(cfg_small(0)) as c:
        assert cut_of(c, B, K, N)[:2] == ((128, 1) if N == 11264 else (64, 1))
        y0 = torch.empty((B, N), dtype=torch.bfloat16, device="cuda")
        ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y0)
        torch.cuda.synchronize()
        y, n = torch.empty_like(y0), torch.empty_like(x)
        for _ in range(200):
            ph.photon_rmsnorm(c.h, x, None, 1e-5, n)
            torch.cuda.synchronize()
            ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y)
            torch.cuda.synchronize()
            assert c.status() == 0
            assert torch.equal(y.view(torch.int16), y0.view(torch.int16))


@pytest.mark.parametrize("K,N,cut", [(16384, 2048, (64, 4)), (5632, 4800, (64, 1)), (5632, 4864, (128, 2))])
@pytest.mark.parametrize("B", [1, 16])
def test_linear_of_few_rows_and_a_long_ring(B, K, N, cut):
    """At most 16 rows make the ring's stages smallest, and K turns it several times over, with two MMA warps on alternate stages
    (tiles of 64 columns) and with one: repeated calls give one result, that of torch in 64 bits (half a bf16 step of values
    below 8, and the order of the sums)."""
    x = dev_bf16(wl.normal_bf16(27, "x", (B, K)))
    w = dev_bf16(wl.normal_bf16(27, "w", (K, N), std=K ** -0.5))
    want = x.double() @ w.double()
    with Ctx(cfg_small(0)) as c:
        nt, ks, stages, mma_warps = cut_of(c, B, K, N)
        assert (nt, ks) == cut and mma_warps == (2 if nt == 64 else 1) and K // 64 // ks >= 2 * 2 * stages
        y0, y = (torch.empty((B, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y0)
        for _ in range(40):
            ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y)
            assert c.status() == 0
            assert torch.equal(y.view(torch.int16), y0.view(torch.int16))
    assert (y0.double() - want).abs().max() <= 2.0 ** -6 + 1e-4


@pytest.mark.parametrize("B,K,N", [(1, 64, 64), (17, 192, 128), (33, 1024, 320), (64, 8192, 2048), (127, 2048, 2048), (129, 448, 256),
                                   (256, 5632, 2048), (600, 2048, 3072)])
@pytest.mark.parametrize("out_major", [False, True])
def test_projection_cuts_and_outputs_that_are_only_16_byte_aligned(B, K, N, out_major):
    """One block of K, ragged rows and slices of K; output, residual and bias 16 bytes into their allocations.  Against torch in 64
    bits: half a bf16 step of the result (2^-8 of its magnitude, or of one where it is smaller) and the rounding of sums of K
    products in 32 bits."""
    check_projection(B, K, N, out_major)


# tiles of 64, 128 and 256 columns, unsplit and in clusters of 2 to 8 with even and uneven shares of the columns
CUTS = [(600, 2048, 512, (64, 3)), (33, 2048, 64, (64, 4)), (129, 4096, 4096, (128, 2)), (1, 5632, 3072, (128, 3)), (129, 5632, 2048, (128, 4)),
        (300, 8192, 1024, (128, 5)), (600, 8192, 512, (128, 6)), (1, 8192, 128, (128, 8)), (64, 12224, 128, (128, 8)),
        (1204, 2048, 2048, (256, 1)), (300, 8192, 4096, (256, 2)), (600, 5632, 2048, (256, 3)), (129, 11584, 3072, (256, 4))]


@pytest.mark.parametrize("B,K,N,cut", CUTS)
@pytest.mark.parametrize("out_major", [False, True])
def test_projection_in_every_kind_of_cut(B, K, N, cut, out_major):
    with Ctx(cfg_small(0)) as c:
        assert cut_of(c, B, K, N)[:2] == cut
    check_projection(B, K, N, out_major)


def check_projection(B, K, N, out_major):
    g = torch.Generator("cuda").manual_seed(B + K + N)

    def new(*shape, std=1.0):
        n = int(np.prod(shape))
        return (torch.randn(n + 8, generator=g, device="cuda") * std).to(torch.bfloat16)[8:].view(*shape)

    x, w, bias, res = new(B, K), new(K, N, std=K ** -0.5), new(N), new(B, N)
    want = x.double() @ w.double() + bias.double() + res.double()
    y = new(B, N)
    assert y.data_ptr() % 32 == 16
    with Ctx(cfg_small(0)) as c:
        layout = ph.PHOTON_W_OUT_MAJOR if out_major else ph.PHOTON_W_IN_MAJOR
        ph.photon_linear(c.h, x, w.t().contiguous() if out_major else w, layout, bias, y, residual=res)
        assert c.status() == 0
    assert ((y.double() - want).abs() <= 2.0 ** -8 * want.abs().clamp(min=1.0) + 1e-4).all()


# tiles of 128, 192 and 256 columns for pairs of CTAs: whole, all in halves, the last round in halves; a last tile past N, rows that
# end inside a warp and rows that only the first CTA of a pair has; one block of K, and K that turns the ring
PAIRS = [(1025, 64, 3072, (128, 120, 120)), (1600, 128, 2112, (128, 119, 119)), (1027, 64, 2112, (192, 55, 55)), (4099, 64, 640, (192, 68, 68)),
         (2050, 128, 2112, (192, 74, 124)), (3000, 704, 448, (192, 0, 72)), (1204, 1024, 2048, (192, 55, 55)), (4099, 64, 448, (256, 0, 68)),
         (6000, 192, 1408, (256, 144, 144)), (9001, 64, 2112, (256, 296, 352)), (1990, 2048, 2048, (256, 64, 64))]


@pytest.mark.parametrize("B,K,N,cut", PAIRS)
@pytest.mark.parametrize("out_major", [False, True])
def test_projection_in_every_kind_of_cut_for_pairs(B, K, N, cut, out_major):
    """Bounds as above."""
    with Ctx(cfg_small(0)) as c:
        clusters, out = (ctypes.c_int32 * 9)(), (ctypes.c_int32 * 8)()
        ph.load().photon_internal_clusters(c.h, clusters)
        ph.load().photon_internal_pair_cut(clusters, B, K, N, int(out_major), 1, 0, out)
        assert out[0] and (out[1], out[4], out[5]) == cut
    check_projection(B, K, N, out_major)


@pytest.mark.parametrize("B,K,N", [(1, 2048, 2048), (31, 2048, 2048), (97, 8192, 256), (127, 5632, 2048), (255, 2048, 11264), (1203, 5632, 2048),
                                   (300, 128, 192), (4099, 192, 2816)])
def test_projection_of_rows_that_end_inside_a_warp(B, K, N):
    """Rows past the batch leave a warp's rounds early; the warp-wide instructions that follow must meet it whole.  The
    residual is the output itself, read by live rows only; a guard behind the last row stays as it was."""
    g = torch.Generator("cuda").manual_seed(B)
    x = torch.randn(B, K, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(K, N, generator=g, device="cuda") * K ** -0.5).to(torch.bfloat16)
    buf0 = torch.randn(B + 64, N, generator=g, device="cuda").to(torch.bfloat16)
    want = x.double() @ w.double() + buf0[:B].double()
    with Ctx(cfg_small(0)) as c:
        for _ in range(3):
            buf = buf0.clone()
            ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, buf[:B], residual=buf[:B])
            assert c.status() == 0
            # half a bf16 step, and the rounding of sums of K products in 32 bits
            assert ((buf[:B].double() - want).abs() <= 2.0 ** -8 * want.abs().clamp(min=1.0) + 1e-4).all()
            assert torch.equal(buf[B:].view(torch.int16), buf0[B:].view(torch.int16))


def test_projection_behind_a_line_of_slow_kernels_does_not_count_their_time():
    """Two and a half seconds of kernels that each let the next one start at once, then a projection whose ring is
    refilled: none of its bounded waits (two seconds) may run while the kernels before it do."""
    B, K, N = 16, 8192, 2048
    g = torch.Generator("cuda").manual_seed(3)
    x = torch.randn(B, K, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(K, N, generator=g, device="cuda") * K ** -0.5).to(torch.bfloat16)
    y0, y = (torch.empty((B, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    src = torch.zeros(1 << 31, dtype=torch.int32, device="cuda")                # 8 GiB, read by one CTA at about 90 GB/s
    with Ctx(cfg_small(0)) as c:
        ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y0)
        begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        begin.record()
        for _ in range(28):
            ph.photon_read_probe(c.h, src, ctas=1)
        ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y)
        end.record()
        assert c.status() == 0
        assert begin.elapsed_time(end) > 2100.0, "the line of kernels was shorter than the limit"
    assert torch.equal(y.view(torch.int16), y0.view(torch.int16))


def test_converter_of_a_step_fits_on_an_sm_beside_the_chunk_attention():
    """Inside a step the two run side by side: registers of a CTA of both within the 65,536 of an SM."""
    a, b = ctypes.c_int32(0), ctypes.c_int32(0)
    ph.load().photon_internal_registers(ctypes.byref(a), ctypes.byref(b))
    assert a.value > 0 and b.value > 0 and a.value + b.value <= 65536, (a.value, b.value)


def test_large_tile_kernel_adds_bias_and_residual_and_is_deterministic(oracle):
    """Thousands of rows with bias and a residual that aliases the output; the oracle
    recomputes a sample of rows; two calls give the same bits."""
    B, K, N = 6000, 320, 1792
    x = wl.normal_bf16(24, "x", (B, K))
    w = wl.normal_bf16(24, "w", (K, N), std=K ** -0.5)
    bias, res = wl.normal_bf16(24, "b", (N,), std=0.5), wl.normal_bf16(24, "r", (B, N))
    pick = np.sort(np.random.default_rng(3).choice(B, 200, replace=False))
    pick[0], pick[-1] = 0, B - 1
    want = oracle.linear(x[pick], w, bias, n_threads=NT) + wl.bf16_bits_to_f64(res[pick])
    with Ctx(cfg_small(0)) as c:
        dx, dw, db = dev_bf16(x), dev_bf16(w), dev_bf16(bias)
        y1, y2 = dev_bf16(res).clone(), dev_bf16(res).clone()
        ph.photon_linear(c.h, dx, dw, ph.PHOTON_W_IN_MAJOR, db, y1, residual=y1)
        ph.photon_linear(c.h, dx, dw, ph.PHOTON_W_IN_MAJOR, db, y2, residual=y2)
        assert c.status() == 0
    assert np.array_equal(host_bits(y1), host_bits(y2))
    assert_close(host_f64(y1)[pick], want, "CTA pairs, bias + residual")


def test_linear_one_hot_rows_return_weight_rows_bit_exactly():
    K, N = 4096, 128                                                     # split over a cluster
    w = wl.normal_bf16(23, "w", (K, N))
    x = np.zeros((64, K), np.float32)
    ks = np.arange(64) * 61 % K
    x[np.arange(64), ks] = 1.0
    with Ctx(cfg_small(0)) as c:
        y = torch.empty((64, N), dtype=torch.bfloat16, device="cuda")
        ph.photon_linear(c.h, dev_bf16(wl.f32_to_bf16_bits(x)), dev_bf16(w), ph.PHOTON_W_IN_MAJOR, None, y)
        assert c.status() == 0
    assert np.array_equal(host_bits(y), w[ks])


@pytest.mark.parametrize("idx", [0, 1, 4])
def test_chunker_matches_oracle(oracle, idx):
    """Normalise, then project: the two calls in a row on the workload's shapes."""
    cfg = wl.CONFIGS[idx]
    ci = wl.chunker_inputs(cfg)
    xn_want, want = oracle.chunker(ci["x"], ci["gamma"], ci["eps"], ci["w_in_major"], ci["bias"], n_threads=NT)
    with Ctx(cfg) as c:
        x = dev_bf16(ci["x"])
        xn = torch.empty_like(x)
        y = torch.empty((cfg.B, cfg.D), dtype=torch.bfloat16, device="cuda")
        ph.photon_rmsnorm(c.h, x, dev_bf16(ci["gamma"]), ci["eps"], xn)
        ph.photon_linear(c.h, xn, dev_bf16(ci["w_in_major"]), ph.PHOTON_W_IN_MAJOR, dev_bf16(ci["bias"]), y)
        assert c.status() == 0
    assert_close(host_f64(y), want, f"chunker cfg{idx}")
    assert np.abs(host_f64(xn) - wl.bf16_bits_to_f64(xn_want)).max() <= 2.0 ** -6


def test_bad_arguments_are_refused():
    with Ctx(cfg_small(0)) as c:
        x = torch.zeros((4, 128), dtype=torch.bfloat16, device="cuda")
        w = torch.zeros((128, 64), dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((4, 64), dtype=torch.bfloat16, device="cuda")
        for K, N in [(100, 64), (128, 32), (0, 64)]:
            with pytest.raises(ph.PhotonError) as e:
                ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y, K=K, N=N)
            assert e.value.code == ph.PHOTON_ERR_INVALID_ARG
        with pytest.raises(ph.PhotonError):
            ph.photon_linear(c.h, x, w, 7, None, y)
        with pytest.raises(ph.PhotonError):
            ph.photon_rmsnorm(c.h, x, None, 1e-5, x, cols=12)
        with pytest.raises(ph.PhotonError):
            ph.photon_rmsnorm(c.h, x, None, -1.0, x)
        ph.photon_linear(c.h, x, w, ph.PHOTON_W_IN_MAJOR, None, y, B=0)
        ph.photon_rmsnorm(c.h, x, None, 0.0, x, rows=0)
        assert c.status() == 0
