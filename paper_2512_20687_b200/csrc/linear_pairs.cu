// y = x W + b (+ residual) for batches of hundreds to thousands of rows (the projections and MLP of a decoder layer over
// all in-flight chunks, prefix passes): the case that is bound by the tensor pipe, not by the weight stream.
//
// What bounds it is feeding the tensor cores from the L2: an SM takes in 80-110 KB a microsecond, and a 128 x 256 tile per
// SM wants 48 KB per block of 64 K elements, which its MMAs are through with in 0.27 us.  So two CTAs on neighbouring SMs
// (a cluster, tcgen05 cta_group::2) work on one tile of 256 rows: each brings its own 128 rows of x and half of the
// weight columns, 32 KB, and the pair's tensor cores read both halves.  Each CTA holds its 128 rows of the accumulator.
//
// A pair per two SMs walks over the tiles.  TMEM holds two accumulators of 256 columns: while eight epilogue warps read
// one back (tcgen05.ld, bias, residual, one rounding to bf16, stores of whole sectors), the MMA warp of the first CTA
// already fills the other from the TMA rings, which run on across tile boundaries.  The residual of a tile is requested
// before its accumulator is waited for.  Shared memory per CTA: 6 to 8 stages of one K block of 64 (128 rows of x and up to
// 128 weight columns).  A stage's barrier is the first CTA's: both CTAs' copies are counted there.
//
// Tiles are 256, 192 or 128 columns wide (pair_plan).  The last, partly filled round of tiles is dealt in halves where that
// is shorter.  Columns past N and rows past B read as zero and are not stored.  Every wait is bounded; a wait that
// gives up sets the status bit and a flag that makes every role of its CTA leave its loops.
//
// Measured, us, one CTA per tile of 128 x 256 (before) / pairs: 16384 x 1024 -> 3072 95 / 74, 16384 x 1024 -> 1024 + residual 58 / 36,
// 16384 x 2816 -> 1024 + residual 95 / 69, 16384 x 1024 -> 5632 168 / 130 (1.45 PFLOP/s), 9472 x 4096 -> 2048 129 / 107 (1.48).
// Polling shows here: with sixteen epilogue warps, or eight that poll without a pause, every block of K took 0.37 and 0.30
// us whatever its width; one issuer for weights and x together 0.30.
//
// GATED: the gate/up projection of the MLP with its activation folded in.  The weight is [gate | up] (N = 2F columns); a
// tile takes as many gate columns as up columns of the same features: the first CTA brings the gate half, the second
// the up half, and the epilogue writes silu(g) * u: out [B, F], and the [B, 2F] intermediate never exists.
//
// ROTARY: a fused q/k/v projection that leaves rotated, split and appended (see RopeOut); tiles are whole heads.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"
#include "rope.cuh"

namespace {

constexpr int BM = 128, BK = 64, NT_MAX = 256;      // rows per CTA, K elements per block, widest tile
constexpr int A_BYTES = BM * BK * 2;
constexpr int RING = 196 * 1024, MAX_STAGES = 8;     // 6, 7 or 8 stages of 256, 192 or 128 columns
constexpr int EPI_PARTS = 2, EPI_WARPS = 4 * EPI_PARTS;
constexpr int LL_THREADS = 128 + EPI_WARPS * 32;    // warp 0: weights, warp 1: MMA (owns TMEM), warp 2: x, warps 4..: epilogue
constexpr int LL_SMEM = RING + 1024 + 256;
// ROTARY: a ring of 192 KB, inverse wavelengths (up to 64 doubles), and cosines and sines of up to 64 positions
constexpr int RING_ROTARY = 192 * 1024, INV_AT = RING_ROTARY + 256, TABLE_BYTES = 64 * (64 + 1) * 8;
constexpr int LL_SMEM_ROTARY = RING_ROTARY + 1024 + 256 + 64 * 8 + TABLE_BYTES;
__host__ __device__ constexpr int ring_bytes(bool rotary) { return rotary ? RING_ROTARY : RING; }

enum Epilogue { PLAIN, GATED_MLP, ROTARY };         // what a tile becomes

// How the output is cut: tiles of 256 rows x nt columns; the pieces of a call are `whole` tiles and then the two halves of
// each further tile.
struct PairPlan {
    int nt, m_tiles, n_tiles, whole, pieces;
    int stages, stage_bytes;
    int n_fast;              // tiles of the same rows follow each other
    float us;                // estimate
};

// A tile, or half of one: first row (of the pair), first column (GATED: feature), accumulator columns.
struct Piece {
    int m0, n0, width;
};

template <bool GATED>
__device__ __forceinline__ Piece piece_at(const ConvParams &p, const PairPlan &c, int i) {
    const int t = i < c.whole ? i : c.whole + (i - c.whole) / 2;
    const int m = c.n_fast ? t / c.n_tiles : t % c.m_tiles, n = c.n_fast ? t % c.n_tiles : t / c.m_tiles;
    Piece x{m * 2 * BM, n * c.nt, c.nt};
    if (i >= c.whole) {
        x.width = c.nt / 2;
        x.n0 += (i - c.whole) % 2 * x.width;
    }
    if (GATED) x.n0 /= 2;
    return x;
}

template <bool W_IN_MAJOR, Epilogue EPI>
__global__ void __launch_bounds__(LL_THREADS, 1)
linear_pair_kernel(const ConvParams p, const PairPlan c, const __grid_constant__ CUtensorMap tm_x,
                   const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_w_half) {
    constexpr bool GATED = EPI == GATED_MLP;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;     // (the same in both CTAs)
    uint8_t *gen = smem_raw + (base - ptx::smem_u32(smem_raw));
    constexpr int RING_END = ring_bytes(EPI == ROTARY);
    const uint32_t full = base + RING_END, empty = full + 8 * MAX_STAGES;         // full: the first CTA's are used, for both
    const uint32_t acc_full = empty + 8 * MAX_STAGES, acc_empty = acc_full + 16;   // [2] each; acc_empty: the first CTA's
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(gen + RING_END + 16 * MAX_STAGES + 32);
    volatile int *dead = reinterpret_cast<volatile int *>(gen + RING_END + 16 * MAX_STAGES + 40);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int n_out = GATED ? p.N / 2 : p.N;
    const int n_atoms = p.D / BK, stages = c.stages, stage_bytes = c.stage_bytes;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            ptx::mbar_init(full + 8 * s, 1);
            ptx::mbar_init(empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(acc_full + 8 * b, 1);
            ptx::mbar_init(acc_empty + 8 * b, 2 * EPI_WARPS);   // one arrival per epilogue warp of the pair
        }
        *dead = 0;
        ptx::mbar_fence_init();
        ptx::prefetch_tmap(&tm_x); ptx::prefetch_tmap(&tm_w);
        if (c.pieces > c.whole) ptx::prefetch_tmap(&tm_w_half);
    }
    double *inv = reinterpret_cast<double *>(gen + INV_AT);
    if (EPI == ROTARY && threadIdx.x < p.rope.dh / 2) inv[threadIdx.x] = rope::inverse_wavelength(threadIdx.x, p.rope.dh, p.rope.log2_theta);
    if (warp == 1) ptx::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t *>(tmem_slot)), 2 * NT_MAX);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();                        // the barriers that the other CTA's copies and arrivals go to exist
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    ptx::grid_dep_launch();

    auto give_up = [&]() { atomicOr(p.status, PHOTON_DEV_TIMEOUT); *dead = 1; };

    if (warp == 0 || warp == 2) {
        // ---- producers, of weights and of x (an issuer's wait and copies take as long as a narrow tile's MMAs): the ring
        // runs on across piece boundaries.  Weights that may be read ahead of the dependency wait fill the ring's first turn there.
        if (ptx::elect_one()) {
            const bool weights = warp == 0;
            const uint32_t full0 = ptx::map_cluster(full, 0);
            bool waited = !weights || !p.w_ahead;
            if (waited) ptx::grid_dep_wait();
            int st = 0, s = 0;
            uint32_t phase = 0;
            for (int i = pair; i < c.pieces && !*dead; i += pairs) {
                const Piece x = piece_at<GATED>(p, c, i);
                const int own = x.width / 2, col = GATED ? rank * n_out + x.n0 : x.n0 + rank * own, row = x.m0 + rank * BM;
                const bool two = own > 64;                                      // N-major: boxes of 64 columns
                const uint32_t bytes = 2 * (A_BYTES + (W_IN_MAJOR ? (two ? 2 : 1) * BK * 128 : own * 128));
                const CUtensorMap *tw = !W_IN_MAJOR && i >= c.whole ? &tm_w_half : &tm_w;
                for (int a = 0; a < n_atoms; ++a, ++st) {
                    if (st >= stages) {
                        // no stage comes free before the dependency is over, and the limit of a wait must not count the kernel before
                        if (!waited) { ptx::grid_dep_wait(); waited = true; }
                        if (!ptx::mbar_wait(empty + 8 * s, phase ^ 1)) { give_up(); break; }
                    }
                    const uint32_t at = base + s * stage_bytes, bar = full0 + 8 * s;
                    if (weights) {
                        if (rank == 0) ptx::mbar_arrive_expect_tx(full + 8 * s, bytes);
                        if (W_IN_MAJOR) {
                            ptx::tma_load_2d_pair(at + A_BYTES, &tm_w, col, a * BK, bar);
                            if (two) ptx::tma_load_2d_pair(at + A_BYTES + BK * 128, &tm_w, col + 64, a * BK, bar);
                        } else {
                            ptx::tma_load_2d_pair(at + A_BYTES, tw, a * BK, col, bar);
                        }
                    } else {
                        ptx::tma_load_2d_pair(at, &tm_x, a * BK, row, bar);
                    }
                    if (++s == stages) { s = 0; phase ^= 1; }
                }
            }
            if (!waited) ptx::grid_dep_wait();
            // the copies of the last turn have landed, and the pair's MMAs have read them, before this CTA leaves
            for (int j = 0; j < stages && j < st; ++j) {
                const int at = st - 1 - j;
                if (!ptx::mbar_wait(empty + 8 * (at % stages), (at / stages) & 1, *dead ? 20000000ull : 2000000000ull)) give_up();
            }
        }
    } else if (warp == 1) {
        // ---- MMA, by the first CTA for both: piece i of this pair accumulates into buffer i & 1 ----
        if (rank == 0 && ptx::elect_one()) {
            ptx::grid_dep_wait();               // (the limit of its waits must not count the kernels before this one)
            int s = 0, n = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int i = pair; i < c.pieces && ok && !*dead; i += pairs, ++n) {
                const int buf = n & 1;
                const Piece x = piece_at<GATED>(p, c, i);
                const uint32_t idesc = ptx::umma_idesc_bf16(2 * BM, x.width, false, W_IN_MAJOR);
                if (!ptx::mbar_wait_cluster(acc_empty + 8 * buf, ((n >> 1) & 1) ^ 1)) { give_up(); break; }
                ptx::tc_fence_after();
                const uint32_t acc = tmem + buf * NT_MAX;
                for (int a = 0; a < n_atoms; ++a) {
                    if (!ptx::mbar_wait(full + 8 * s, phase)) { give_up(); ok = false; break; }
                    ptx::tc_fence_after();
                    const uint32_t a_addr = base + s * stage_bytes, b_addr = a_addr + A_BYTES;
                    const uint64_t adesc = ptx::umma_desc_sw128(a_addr, 0, 1024);
                    const uint64_t bdesc = ptx::umma_desc_sw128(b_addr, W_IN_MAJOR ? BK * 128 : 0, 1024);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        ptx::umma_bf16_pair(acc, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(W_IN_MAJOR ? k * 128 : k * 2), idesc,
                                            (a | k) != 0);
                    ptx::umma_commit_pair(empty + 8 * s);                       // frees the stage in both CTAs
                    if (a == n_atoms - 1) ptx::umma_commit_pair(acc_full + 8 * buf);
                    if (++s == stages) { s = 0; phase ^= 1; }
                }
            }
        }
    } else if (warp >= 4) {
        // ---- epilogue: warp w reads TMEM lanes [32*(w%4), +32) = rows of this CTA, every other group of 32 columns ----
        ptx::grid_dep_wait();
        const int quad = warp & 3, part = (warp - 4) >> 2;
        const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t acc_empty0 = ptx::map_cluster(acc_empty, 0);
        const bool wide = (reinterpret_cast<uintptr_t>(p.U) & 31u) == 0;
        auto store = [&](bf16 *dst, const uint32_t *w) {                       // 16 columns
            if (wide) { ptx::stg256(dst, w); return; }
            *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(dst + 8) = make_uint4(w[4], w[5], w[6], w[7]);
        };
        [[maybe_unused]] rope::Table angles{reinterpret_cast<float2 *>(inv + 64), inv, rope::positions(p.rope), p.rope.dh / 2, rope::table_stride(p.rope.dh)};
        if constexpr (EPI == ROTARY) {
            angles.fill(threadIdx.x - 128, 32 * EPI_WARPS);
            ptx::named_bar_sync(1, 32 * EPI_WARPS);
        }
        int n = 0;
        for (int i = pair; i < c.pieces && !*dead; i += pairs, ++n) {
            const int buf = n & 1;
            const Piece x = piece_at<GATED>(p, c, i);
            const int b = x.m0 + rank * BM + quad * 32 + lane;
            const bool live = b < p.B;
            constexpr int ROUNDS = NT_MAX / (32 * EPI_PARTS);                   // groups of 32 columns per warp, at most
            [[maybe_unused]] uint4 res[EPI == PLAIN ? ROUNDS : 1][4];
            if constexpr (EPI == PLAIN) {
                if (p.residual && live) {
                    const bf16 *row = p.residual + (size_t)b * p.N + x.n0;
#pragma unroll
                    for (int j = 0; j < ROUNDS; ++j) {
                        const int c0 = 32 * (part + EPI_PARTS * j);
                        if (c0 < x.width && x.n0 + c0 < n_out)
#pragma unroll
                            for (int v = 0; v < 4; ++v) res[j][v] = __ldcg(reinterpret_cast<const uint4 *>(row + c0) + v);
                    }
                }
            }
            [[maybe_unused]] rope::Row to;
            if (EPI == ROTARY && live) to = rope::Row(p.rope, b);
            // one lane polls, and not all the time: polling takes issue slots and barrier accesses from the warps that feed the MMAs
            bool ok = lane != 0 || ptx::mbar_wait_idle(acc_full + 8 * buf, (n >> 1) & 1);
            ok = __shfl_sync(0xffffffffu, (int)ok, 0);
            if (!ok) { if (lane == 0) give_up(); break; }
            ptx::tc_fence_after();
            if constexpr (GATED) {
                // 16 features at a time: their gate columns, and their up columns half a piece further on
#pragma unroll 1
                for (int f = 16 * part; f < x.width / 2; f += 16 * EPI_PARTS) {
                    uint32_t g[16], u[16], w[8];
                    __syncwarp();                                               // rows past the batch skip the stores of the round before
                    ptx::tmem_ld_32x16(lanes + buf * NT_MAX + f, g);
                    ptx::tmem_ld_32x16(lanes + buf * NT_MAX + x.width / 2 + f, u);
                    ptx::tmem_ld_wait();
                    if (!live || x.n0 + f >= n_out) continue;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        // the projections are rounded to bf16 first, as when they are stored and read back
                        const float g0 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(g[2 * e])));
                        const float g1 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(g[2 * e + 1])));
                        const float u0 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(u[2 * e])));
                        const float u1 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(u[2 * e + 1])));
                        const __nv_bfloat162 o = __floats2bfloat162_rn(g0 / (1.f + __expf(-g0)) * u0, g1 / (1.f + __expf(-g1)) * u1);
                        w[e] = *reinterpret_cast<const uint32_t *>(&o);
                    }
                    store(p.U + (size_t)b * n_out + x.n0 + f, w);
                }
            } else if constexpr (EPI == ROTARY) {
                // 16 feature pairs at a time, for all heads of the piece: their angles are the same
                const int dh = p.rope.dh;
#pragma unroll 1
                for (int j = 16 * part; j < dh / 2; j += 16 * EPI_PARTS) {
                    float cs[16], sn[16];
                    angles.get(to.at, j, cs, sn);
                    int h = x.n0 / dh;
#pragma unroll 1
                    for (int c0 = 0; c0 < x.width; c0 += dh, ++h) {
                        uint32_t lo[16], hi[16];
                        __syncwarp();                                           // (likewise)
                        ptx::tmem_ld_32x16(lanes + buf * NT_MAX + c0 + j, lo);
                        ptx::tmem_ld_32x16(lanes + buf * NT_MAX + c0 + dh / 2 + j, hi);
                        ptx::tmem_ld_wait();
                        if (live && x.n0 + c0 < n_out) rope::store<16>(p.rope, to, h, j, lo, hi, cs, sn);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < ROUNDS; ++j) {
                    const int c0 = 32 * (part + EPI_PARTS * j);
                    if (c0 >= x.width || x.n0 + c0 >= n_out) break;             // (N is a multiple of 64, widths of 32)
                    uint32_t r[32], w[16];
                    __syncwarp();                                               // (likewise)
                    ptx::tmem_ld_32x32(lanes + buf * NT_MAX + c0, r);
                    ptx::tmem_ld_wait();
                    if (live) {
                        const int col = x.n0 + c0;
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            uint4 rv = make_uint4(0u, 0u, 0u, 0u), bv = rv;
                            if (p.residual) rv = res[j][v];
                            if (p.bias) bv = __ldcg(reinterpret_cast<const uint4 *>(p.bias + col) + v);
                            const uint32_t rw[4] = {rv.x, rv.y, rv.z, rv.w}, bw[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float f0 = __uint_as_float(r[v * 8 + 2 * e]) + bf16_lo(rw[e]) + bf16_lo(bw[e]);
                                const float f1 = __uint_as_float(r[v * 8 + 2 * e + 1]) + bf16_hi(rw[e]) + bf16_hi(bw[e]);
                                const __nv_bfloat162 o = __floats2bfloat162_rn(f0, f1);
                                w[v * 4 + e] = *reinterpret_cast<const uint32_t *>(&o);
                            }
                        }
                        bf16 *dst = p.U + (size_t)b * p.N + col;
                        store(dst, w);
                        store(dst + 16, w + 8);
                    }
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(acc_empty0 + 8 * buf);     // the MMA warp may overwrite this buffer
        }
    }
    __syncwarp();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();                        // neither CTA leaves while the other may still signal it or read its ring
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc_pair(tmem, 2 * NT_MAX);
    }
}

// The cut with the least estimated time (microseconds), from 800 timed calls (8 weight shapes, 129 to 8192 rows, every width with
// and without halves, weights and x out of the HBM).  A block of 64 K elements takes 0.27 to 0.33 at 256 columns, where the
// MMAs (512 cycles) and 32 KB from the L2 cost the same, 0.225 at 192, and 0.21 below, where the latency of a stage's copies shows;
// a round of tiles whose epilogue overlaps the next costs 1.2 more, the call's start and its last epilogue 4 to 5.6.  The cut it
// takes is 2 % slower than the fastest on average.  1204 x 5632 -> 2048: 28.4 us as 55 tiles of 192 columns, 35.6 as 40 of 256; 900 x
// 2048 -> 11264: 35.6 with the last round of 28 tiles in halves, 36.9 without.
float block_us(int width) { return width >= 256 ? 0.30f : width >= 192 ? 0.235f : width >= 128 ? 0.215f : 0.21f; }

// grain: what tiles and halves have to be multiples of (0: nothing)
PairPlan pair_plan(int pairs, int B, int K, int N, bool in_major, int grain) {
    PairPlan best{};
    for (int nt = NT_MAX; nt >= 128; nt -= 64) {
        if (grain && nt % grain != 0) continue;
        const int w_cols = in_major ? (nt / 2 + 63) / 64 * 64 : nt / 2;     // N-major weights come in boxes of 64 columns
        const int stage_bytes = A_BYTES + w_cols * BK * 2, atoms = K / BK;
        PairPlan c{nt, (B + 2 * BM - 1) / (2 * BM), (N + nt - 1) / nt, 0, 0, std::min(MAX_STAGES, ring_bytes(grain > 0) / stage_bytes), stage_bytes, 0, 0.f};
        const int tiles = c.m_tiles * c.n_tiles, rounds = tiles / pairs, rest = tiles % pairs;
        const bool halves = rest > 0 && 2 * rest <= pairs && !(grain && nt / 2 % grain != 0);
        const int last = rest == 0 || (halves && rounds > 0) ? nt : halves ? nt / 2 : nt;
        c.us = rounds * (atoms * block_us(nt) + 1.2f) + (rest ? atoms * block_us(halves ? nt / 2 : nt) : 0.f) +
               (last >= 256 ? 5.6f : last >= 192 ? 4.9f : 4.1f);
        c.whole = halves ? tiles - rest : tiles;
        c.pieces = c.whole + 2 * (tiles - c.whole);
        c.n_fast = N <= B;                                                 // the smaller operand stays in the L2
        if (best.nt == 0 || c.us < best.us) best = c;
    }
    return best;
}

int grain_of(const ConvParams &p) { return p.rope.q ? p.rope.dh : 0; }

template <bool IN_MAJOR, Epilogue EPI>
cudaError_t run_large(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    static size_t smem_set[kMaxDevices] = {};
    constexpr size_t smem = EPI == ROTARY ? LL_SMEM_ROTARY : LL_SMEM;
    if (const cudaError_t e = ensure_dynamic_smem(linear_pair_kernel<IN_MAJOR, EPI>, smem, ctx->device, smem_set)) return e;
    if (p.B == 0) return cudaSuccess;
    const int pairs = ctx->clusters[2];
    const PairPlan c = pair_plan(pairs, p.B, p.D, p.N, IN_MAJOR, grain_of(p));
    const CUtensorMap *t;
    CUtensorMap mx, mw, mw_half;
    if (!(t = ctx->tmaps.get(p.x, (uint64_t)p.B, (uint64_t)p.D, BM))) return cudaErrorInvalidValue;
    mx = *t;
    if (IN_MAJOR) t = ctx->tmaps.get(p.w, (uint64_t)p.D, (uint64_t)p.N, BK);        // [K, N], boxes of 64 k x 64 n
    else t = ctx->tmaps.get(p.w, (uint64_t)p.N, (uint64_t)p.D, c.nt / 2);           // [N, K], boxes of nt/2 n x 64 k, and half of that
    if (!t) return cudaErrorInvalidValue;
    mw = mw_half = *t;
    if (!IN_MAJOR && c.pieces > c.whole) {
        if (!(t = ctx->tmaps.get(p.w, (uint64_t)p.N, (uint64_t)p.D, c.nt / 4))) return cudaErrorInvalidValue;
        mw_half = *t;
    }
    const cudaError_t e = launch_dependent(linear_pair_kernel<IN_MAJOR, EPI>, dim3(2 * std::min(c.pieces, pairs)),
                                           dim3(LL_THREADS), smem, st, 2, p, c, mx, mw, mw_half);
    ++*launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Where the pair kernel is the faster one, by both kernels' estimates; the pairs' is a little low.  us, projection kernel / pairs:
// 700 x 2048 -> 3072 11.7 / 12.8, 900 x 2048 -> 3072 16.3 / 14.0, 1204 x 2048 -> 2048 + residual 20.5 / 14.7, 1204 x 1024 -> 1024 8.2 / 8.3,
// 3072 x 1024 -> 1024 15.6 / 11.0, 300 x 2048 -> 11264 18.9 / 22.7, 4096 x 256 -> 512 5.1 / 6.2.  From more than two waves of its largest tiles
// on the projection kernel's estimate is too low, and the pairs are faster wherever it took that kernel (1600 x 2048 -> 8192 49.4 / 44.8,
// out-major 54.3 / 46.8; 3334 x 4096 -> 4096 + residual 99.5 / 87.8, out-major 111.5 / 92.3).
bool linear_wants_pairs(const int *fit, const ConvParams &p, bool gated) {
    if (fit[2] < 1 || p.B <= BM) return false;
    if ((long long)((p.B + 127) / 128) * ((p.N + 255) / 256) > 2ll * fit[1]) return true;
    const float slab = linear_slab_us(fit, p, gated);
    return slab < 0.f || 1.04f * pair_plan(fit[2], p.B, p.D, p.N, !p.w_out_major, grain_of(p)).us < slab;
}

void linear_pair_cut(const int *fit, const ConvParams &p, bool gated, int32_t *cut) {
    const PairPlan c = pair_plan(std::max(1, fit[2]), p.B, p.D, p.N, !p.w_out_major, grain_of(p));
    const int32_t v[] = {linear_wants_pairs(fit, p, gated), c.nt, c.m_tiles, c.n_tiles, c.whole, c.pieces, c.stages, c.stage_bytes};
    std::copy(v, v + 8, cut);
}

cudaError_t launch_linear_pairs(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return p.w_out_major ? run_large<false, PLAIN>(ctx, p, st, launches) : run_large<true, PLAIN>(ctx, p, st, launches);
}

cudaError_t launch_qkv_rope_pairs(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return p.w_out_major ? run_large<false, ROTARY>(ctx, p, st, launches) : run_large<true, ROTARY>(ctx, p, st, launches);
}

// out [B, F] = silu(x Wg) * (x Wu) for w = [Wg | Wu] with N = 2F columns; for the shapes
// linear_wants_pairs accepts.  No bias, no residual.
cudaError_t launch_gate_up_pairs(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return p.w_out_major ? run_large<false, GATED_MLP>(ctx, p, st, launches) : run_large<true, GATED_MLP>(ctx, p, st, launches);
}
