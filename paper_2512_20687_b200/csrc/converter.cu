// Context converter U^(l) (Section 2.1.2): U[b, n] = sum_k x[b,k] W[k,n] (+ bias[n]),
// n = r*D + j for prefix r, feature j; and every other projection y = x W (+ b) (+ residual)
// of up to some hundreds of rows (K and N multiples of 64): the context chunker's, the layers'.
//
// At these sizes the weights are most of what is read, so the kernel is built around their stream.
// The output is cut into tiles of 128 batch rows x NT weight columns, and the K range of a tile over
// a thread-block cluster of ksplit CTAs, so that about every SM holds a CTA with an equal share of the
// weights (the launcher's rule is beside it).  A CTA has a TMA ring whose stages hold one or two blocks of 64
// K elements: of the NT weight columns, and of the x rows the batch needs.  Weights and x are issued by a
// warp each.  Where the projection follows another kernel of the same call (w_ahead), the weight half of the
// whole ring is requested before the dependency wait: the kernel before does not write weights, and it lets
// this one start only after its own wait, when everything before the call has been written.  A call that begins with
// a projection waits first: its weights may be what the call before it writes.  The contraction is tcgen05.mma (batch rows on the M side, fp32 in
// TMEM); an MMA spans 128 rows, what it reads beyond the fetched ones only reaches accumulator rows that
// nobody reads.
//
// A split tile is put together by reduce-scatter: the tile's columns are dealt to the CTAs of the
// cluster in groups of 16; every CTA stages the groups of the others in its (by then free) ring, one
// bulk copy per peer moves them through distributed shared memory, and each CTA adds what it received
// to its own groups in rank order (the result does not depend on timing), adds bias and residual,
// rounds once and stores.
//
// GATED: the gate/up projection of the MLP with its activation folded in.  W is [gate | up] with N = 2F
// columns; a tile is NT/2 gate columns and the NT/2 up columns of the same features, and silu(gate) * up goes
// into U [B, F] (both rounded to bf16 first, as when they are stored and read back by the activation
// kernel).  No bias, no residual.
//
// ROTARY: a fused q/k/v projection that leaves rotated, split and appended (see RopeOut).  A tile is one head; a group of columns is 8
// features and their rotation partners.  Cosines and sines of the first positions (31 of heads of 128, 62 of 64) come from a table that
// four warps fill under the contraction; those of later positions are computed where they are used.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "rope.cuh"

namespace {

constexpr int BM = 128;                 // batch rows per tile (UMMA M)
constexpr int BK = 64;                  // K elements per block (one 128-byte swizzled row)
constexpr int SLAB_THREADS = 256;       // warp 0: weights, 1 and 7: MMA (1 owns TMEM), 6: x; then all eight: epilogue
// Blocks per stage.  A stage costs its issuers and the MMA warp a round trip to a barrier (95 cycles) and more beside
// the copies and MMAs themselves (48 to 64 cycles each for narrow tiles): with one block per stage that paced tiles of 64
// columns at 200 ns per block, whatever was loaded.
__host__ __device__ constexpr int blocks_per_stage(int nt) { return nt <= 128 ? 2 : 1; }
// Tiles of 64 columns have two MMA warps, on alternate stages and with an accumulator each (the epilogue adds them), so that
// one's barrier and commit (36 cycles) pass under the other's MMAs: with one, the drain of a ring that was filled ahead of the
// dependency wait is 1.2 us longer (converter of 64 rows, 2048 -> 8192, inside the decode step).  The stages are then a
// multiple of the MMA warps: each warp meets every phase of the barriers it waits for.
__host__ __device__ constexpr int mma_warps(int nt) { return nt == 64 ? 2 : 1; }
// Tiles of 64 columns are what a decode step's converter runs on, beside the chunk attention, whose CTAs hold up to 43,008
// registers: 80 per thread (20,480) leave room for one on the SM, the 146 that two groups of columns at a time take (38,912)
// have the converter wait until its SMs are empty (64 sequences, step replayed 28.5 -> 27.8 us, called one by one 33.7 -> 31.4).
__host__ __device__ constexpr int groups_at_once(int nt) { return nt == 64 ? 1 : 2; }
__host__ __device__ constexpr int min_ctas(int nt) { return nt == 64 ? 3 : 1; }     // (of registers; shared memory holds one)
constexpr int MAX_STAGES = 12;
constexpr int GROUP = 16;               // accumulator columns that change hands together
constexpr int QUAD_BYTES = 32 * GROUP * 4;          // a group's values of 32 rows
constexpr int BAR_BYTES = 512;
constexpr int RING_BYTES = 208 * 1024;
constexpr int ANGLES_BYTES = 16 * 1024;             // ROTARY: cosines and sines of the first positions

// First group of the part of a tile that CTA r of ks puts together.
__host__ __device__ __forceinline__ int first_group(int groups, int r, int ks) { return groups * r / ks; }

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&t);
}

enum Epilogue { PLAIN, GATED_MLP, ROTARY };     // what a tile becomes

// n groups of this warp's 32 rows from the accumulator (both: the sum of two).  HALVES: group g is 8 columns of the tile's first half
// and the 8 of its second half that belong to them (gate and up columns of the same features; a feature and its rotation partner).
template <int NT, bool HALVES, int n>
__device__ __forceinline__ void load_groups(uint32_t acc, bool both, int g, uint32_t (&r)[n * GROUP]) {
    auto load = [&](uint32_t from, uint32_t *to) {
#pragma unroll
        for (int h = 0; h < n; ++h) {
            if constexpr (HALVES) {
                ptx::tmem_ld_32x8(from + (g + h) * (GROUP / 2), to + h * GROUP);
                ptx::tmem_ld_32x8(from + NT / 2 + (g + h) * (GROUP / 2), to + h * GROUP + GROUP / 2);
            } else {
                ptx::tmem_ld_32x16(from + (g + h) * GROUP, to + h * GROUP);
            }
        }
    };
    load(acc, r);
    if constexpr (mma_warps(NT) == 2) {
        uint32_t r2[n * GROUP];
        load(acc + NT, r2);
        ptx::tmem_ld_wait();
        if (both)
#pragma unroll
            for (int e = 0; e < n * GROUP; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(r2[e]));
    } else {
        ptx::tmem_ld_wait();
    }
}

template <int NT, bool W_IN_MAJOR, Epilogue EPI>
__global__ void __launch_bounds__(SLAB_THREADS, min_ctas(NT))
linear_slab_kernel(const ConvParams p, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w) {
    constexpr bool GATED = EPI == GATED_MLP, ROPE = EPI == ROTARY, HALVES = EPI != PLAIN;
    constexpr int W_BYTES = NT * BK * 2, GROUPS = NT / GROUP, KA = blocks_per_stage(NT), MW = mma_warps(NT), AT_ONCE = groups_at_once(NT);
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = ptx::smem_u32(smem_raw);
    const int x_bytes = p.x_rows * BK * 2;
    const uint32_t w_base = base + p.stages * KA * x_bytes;      // all x blocks first: an MMA reads past the end of a short one
    const uint32_t full = base + RING_BYTES, empty = full + 8 * MAX_STAGES;
    const uint32_t bar_acc = empty + 8 * MAX_STAGES, bar_rx = bar_acc + 8;   // accumulator complete; peers' groups landed
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem_raw + RING_BYTES + 16 * MAX_STAGES + 16);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ks = p.ksplit, zr = (int)(blockIdx.x % ks);        // zr = rank in the cluster: which slice of K
    const int n0 = (int)(blockIdx.x / ks) * (GATED ? NT / 2 : NT), m0 = blockIdx.y * BM;
    const int up0 = p.N / 2 + n0;                                // GATED: first of this tile's up columns
    const int a_lo = (p.D / BK) * zr / ks, n_atoms = (p.D / BK) * (zr + 1) / ks - a_lo;
    const int n_steps = (n_atoms + KA - 1) / KA;
    const int nq = p.x_rows > 32 ? p.x_rows / 32 : 1;            // quarters of the tile's rows that hold batch rows
    const int g_lo = first_group(GROUPS, zr, ks), own = first_group(GROUPS, zr + 1, ks) - g_lo;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            ptx::mbar_init(full + 8 * s, p.once ? 1 : 2);        // an arrival per issuer, each with its own bytes
            ptx::mbar_init(empty + 8 * s, 1);
        }
        ptx::mbar_init(bar_acc, MW);
        ptx::mbar_init(bar_rx, 1);
        ptx::mbar_fence_init();
        if (ks > 1) ptx::mbar_arrive_expect_tx(bar_rx, (ks - 1) * own * nq * QUAD_BYTES);
        ptx::prefetch_tmap(&tm_x); ptx::prefetch_tmap(&tm_w);
    }
    double *inv = reinterpret_cast<double *>(smem_raw + RING_BYTES + BAR_BYTES);   // ROPE: a tile is one head, dh = NT
    [[maybe_unused]] rope::Table angles{reinterpret_cast<float2 *>(inv + NT / 2), inv,
                                        min(p.rope.period, ANGLES_BYTES / (rope::table_stride(NT) * 8)), NT / 2, rope::table_stride(NT)};
    if (ROPE && threadIdx.x < NT / 2) inv[threadIdx.x] = rope::inverse_wavelength(threadIdx.x, NT, p.rope.log2_theta);
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t *>(tmem_slot)), MW * NT);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    ptx::grid_dep_launch();

    // One lane of each of these warps does the work; there is nothing to vote on.  A ring that is filled once, its weights ahead
    // of the wait, is filled by one thread: a second issuer costs such short calls 0.2 us (64 x 256 -> 256: 2.9 and 2.6 us).  In
    // longer ones, or with the weights behind the wait too, the second is worth having (16 x 1024 -> 1024, all behind the wait: 4.9
    // and 4.6 us).
    auto load_x = [&](int st, int s, int n) {                    // x[m0.., k0..]
#pragma unroll
        for (int j = 0; j < KA; ++j)
            if (j < n) ptx::tma_load_2d(base + (s * KA + j) * x_bytes, &tm_x, (a_lo + st * KA + j) * BK, m0, full + 8 * s);
    };
    auto load_w = [&](int st, int s, int n) {
#pragma unroll
        for (int j = 0; j < KA; ++j) {
            if (j >= n) break;
            const int k0 = (a_lo + st * KA + j) * BK;
            const uint32_t dst = w_base + (s * KA + j) * W_BYTES, bar = full + 8 * s;
            if (!W_IN_MAJOR) {
                ptx::tma_load_2d(dst, &tm_w, k0, n0, bar);                               // W[n0.., k0..]  (K-major)
                if (GATED) ptx::tma_load_2d(dst + W_BYTES / 2, &tm_w, k0, up0, bar);
            } else {
#pragma unroll
                for (int jj = 0; jj < NT / 64; ++jj)                                     // W[k0.., n..] (N-major), 64 columns a box
                    ptx::tma_load_2d(dst + jj * (BK * 128), &tm_w,
                                     GATED ? (jj < NT / 128 ? n0 + 64 * jj : up0 + 64 * (jj - NT / 128)) : n0 + 64 * jj, k0, bar);
            }
        }
    };
    if (warp != 0 || !p.w_ahead) ptx::grid_dep_wait();           // x may be the output of the kernel before this one
    if (p.once) {
        if (warp == 0 && ptx::elect_one()) {
            for (int st = 0; st < n_steps; ++st) {
                const int n = min(KA, n_atoms - st * KA);
                ptx::mbar_arrive_expect_tx(full + 8 * st, n * (x_bytes + W_BYTES));
                load_w(st, st, n);
            }
            ptx::grid_dep_wait();
            for (int st = 0; st < n_steps; ++st) load_x(st, st, min(KA, n_atoms - st * KA));
        }
    } else if ((warp == 0 || warp == 6) && ptx::elect_one()) {
        int s = 0;
        for (int st = 0; st < n_steps; ++st) {
            // no stage comes free before the dependency is over, and the limit of a wait must not count the kernel before
            if (st == p.stages && warp == 0) ptx::grid_dep_wait();
            if (st >= p.stages && !ptx::mbar_wait(empty + 8 * s, (st / p.stages - 1) & 1)) {
                atomicOr(p.status, PHOTON_DEV_TIMEOUT);
                break;
            }
            const int n = min(KA, n_atoms - st * KA);
            ptx::mbar_arrive_expect_tx(full + 8 * s, n * (warp == 6 ? x_bytes : W_BYTES));
            if (warp == 6) load_x(st, s, n);
            else load_w(st, s, n);
            if (++s == p.stages) s = 0;
        }
    }
    if ((warp == 1 || (MW == 2 && warp == 7)) && ptx::elect_one()) {
        constexpr uint32_t idesc = ptx::umma_idesc_bf16(BM, NT, false, W_IN_MAJOR);
        const int me = warp == 1 ? 0 : 1;                        // which stages, which accumulator
        int s = me;
        uint32_t phase = 0;
        if (me >= n_steps) ptx::mbar_arrive(bar_acc);            // fewer steps than MMA warps
        for (int st = me; st < n_steps; st += MW) {
            if (!ptx::mbar_wait(full + 8 * s, phase)) {
                atomicOr(p.status, PHOTON_DEV_TIMEOUT);
                break;
            }
            const int n = min(KA, n_atoms - st * KA);
#pragma unroll
            for (int j = 0; j < KA; ++j) {
                if (j >= n) break;
                const uint64_t adesc = ptx::umma_desc_sw128(base + (s * KA + j) * x_bytes, 0, 1024);
                const uint64_t bdesc = ptx::umma_desc_sw128(w_base + (s * KA + j) * W_BYTES, W_IN_MAJOR ? BK * 128 : 0, 1024);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    // advance 16 K elements: 32 bytes inside the swizzled row (K-major),
                    // 16 rows of 128 bytes (N-major); the address field counts 16-byte units
                    ptx::umma_bf16(tmem + me * NT, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(W_IN_MAJOR ? k * 128 : k * 2), idesc,
                                   st != me || (j | k) != 0);
            }
            ptx::umma_commit(st + MW >= n_steps ? bar_acc : empty + 8 * s); // frees the stage once these MMAs have read it
            s += MW;
            if (s >= p.stages) { s -= p.stages; phase ^= 1; }
        }
    }
    if (ROPE && warp >= 2 && warp < 6) angles.fill(threadIdx.x - 64, 128);
    __syncwarp();
    if (ROPE) __syncthreads();

    if (warp == 0) ptx::grid_dep_wait();                         // (the weights did not wait; what follows does)

    // ---- epilogue: warp w reads TMEM lanes [32*(w%4), +32) = batch rows m0 + that range, half of the groups each:
    // one warp per scheduler is bound by the latency of its own instructions, so all eight take part
    const int quad = warp & 3, half = warp >> 2;
    const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16);
    const bool both = n_steps > 1;          // (with one step the second accumulator is untouched)
    const int b = m0 + quad * 32 + lane;
    const bool live = quad < nq && b < p.B;
    const int mid = g_lo + (own + 1) / 2;   // groups [g_lo, mid) are the first four warps', the rest the others'
    const int g_begin = half ? mid : g_lo, g_end = half ? g_lo + own : mid;
    // the residual of the next groups to finish, requested well before it is added: a trip to the L2 per round otherwise
    // (4096 x 2048 -> 2048: 46.9 us, 42 since)
    uint4 res[AT_ONCE * GROUP / 8];
    auto fetch_residual = [&](int g) {
        if constexpr (EPI == PLAIN) {
            if (!p.residual || !live) return;
#pragma unroll
            for (int v = 0; v < AT_ONCE * GROUP / 8; ++v)
                if (g + v / (GROUP / 8) < g_end)
                    res[v] = __ldcg(reinterpret_cast<const uint4 *>(p.residual + (size_t)b * p.N + n0 + g * GROUP) + v);
        }
    };
    fetch_residual(g_begin);
    [[maybe_unused]] const rope::Row to = [&]() {
        if (ROPE && live) return rope::Row(p.rope, b);
        return rope::Row();
    }();
    // one lane polls: 256 threads at the barrier hold up those that feed it (128 x 1024 -> 1024: 5.2 us, 5.0 with one)
    bool ok = lane != 0 || ptx::mbar_wait(bar_acc, 0);
    if (!ok) atomicOr(p.status, PHOTON_DEV_TIMEOUT);
    ok = __shfl_sync(0xffffffffu, (int)ok, 0);
    __syncwarp();
    ptx::tc_fence_after();
    const uint32_t recv = base + (GROUPS - GROUPS / ks) * nq * QUAD_BYTES;       // behind the largest staging area of any rank
    if (ks > 1) {
        ptx::cluster_arrive();                             // this CTA's ring is free
        if (quad < nq)
            for (int g = AT_ONCE * half; g < GROUPS; g += 2 * AT_ONCE) {   // the other CTAs' groups, in the order of their owners
                uint32_t r[AT_ONCE * GROUP];
                load_groups<NT, HALVES, AT_ONCE>(acc, both, g, r);
#pragma unroll
                for (int h = 0; h < AT_ONCE; ++h) {
                    if (g + h >= g_lo && g + h < g_lo + own) continue;
                    const uint32_t at = base + ((g + h < g_lo ? g + h : g + h - own) * nq + quad) * QUAD_BYTES + lane * 16;
#pragma unroll
                    for (int j = 0; j < GROUP / 4; ++j)
                        ptx::sts128(at + j * 512, make_uint4(r[GROUP * h + 4 * j], r[GROUP * h + 4 * j + 1], r[GROUP * h + 4 * j + 2],
                                                             r[GROUP * h + 4 * j + 3]));
                }
            }
        ptx::fence_proxy_async();                          // the staged groups are read by bulk copies
        __syncthreads();
        ptx::cluster_wait();                               // every CTA's ring is free: groups may land there
        if (warp == 2 && lane < ks && lane != zr) {
            // lane -> peer: its groups of this CTA's tile, to the place of this rank in the peer's receive area
            const int lo = first_group(GROUPS, lane, ks), cnt = first_group(GROUPS, lane + 1, ks) - lo;
            const uint32_t bytes = cnt * nq * QUAD_BYTES;
            ptx::bulk_copy_to_peer(ptx::map_cluster(recv + (zr < lane ? zr : zr - 1) * bytes, lane),
                                   base + (lo < g_lo ? lo : lo - own) * nq * QUAD_BYTES, bytes, ptx::map_cluster(bar_rx, lane));
        }
        __syncwarp();
    }
    if (quad < nq) {
        int g = g_begin;
        // whole sectors where the output's alignment allows it (16 bytes are all that the caller owes, and a gated pair
        // that starts at an odd group starts in the middle of a sector)
        const bool wide = (reinterpret_cast<uintptr_t>(p.U) & 31u) == 0 && !(GATED && (g & 1));
        if (ks > 1) {
            const bool got = __all_sync(0xffffffffu, ptx::mbar_wait(bar_rx, 0));
            if (!got && lane == 0) atomicOr(p.status, PHOTON_DEV_TIMEOUT);
            ok = ok && got;
        }
        // groups [g, g + n): own accumulator + the other slices in rank order, then bias, residual, rounding
        auto finish = [&](auto n_tag, int g) {
            constexpr int n = decltype(n_tag)::value, COLS = n * GROUP, WORDS = GATED ? COLS / 4 : COLS / 2;
            uint32_t r[COLS], w[WORDS];
            [[maybe_unused]] const int col = n0 + g * GROUP;
            __syncwarp();                                  // rows past the batch took no part above, and left the round before early
            load_groups<NT, HALVES, n>(acc, both, g, r);
            for (int z = 0; z < ks - 1; ++z)
#pragma unroll
                for (int h = 0; h < n; ++h) {
                    const uint32_t at = recv + ((z * own + g + h - g_lo) * nq + quad) * QUAD_BYTES + lane * 16;
#pragma unroll
                    for (int j = 0; j < GROUP / 4; ++j) {
                        const uint4 v = ptx::lds128(at + j * 512);
                        uint32_t *d = r + h * GROUP + 4 * j;
                        d[0] = __float_as_uint(__uint_as_float(d[0]) + __uint_as_float(v.x));
                        d[1] = __float_as_uint(__uint_as_float(d[1]) + __uint_as_float(v.y));
                        d[2] = __float_as_uint(__uint_as_float(d[2]) + __uint_as_float(v.z));
                        d[3] = __float_as_uint(__uint_as_float(d[3]) + __uint_as_float(v.w));
                    }
                }
            if (!live || !ok) return;
            if constexpr (ROPE) {
                constexpr int F = n * GROUP / 2;            // features, and as many partners
                uint32_t lo[F], hi[F];
#pragma unroll
                for (int e = 0; e < F; ++e) {
                    lo[e] = r[e / (GROUP / 2) * GROUP + e % (GROUP / 2)];
                    hi[e] = r[e / (GROUP / 2) * GROUP + GROUP / 2 + e % (GROUP / 2)];
                }
                float cs[F], sn[F];
                angles.get(to.at, g * (GROUP / 2), cs, sn);
                rope::store<F>(p.rope, to, n0 / NT, g * (GROUP / 2), lo, hi, cs, sn);
                return;
            }
            bf16 *dst;
            if constexpr (GATED) {
#pragma unroll
                for (int e = 0; e < WORDS; ++e) {          // group h: 8 gate values, then the 8 up values of the same features
                    const int h = e / (GROUP / 4), i = h * GROUP + 2 * (e % (GROUP / 4));
                    const float g0 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(r[i])));
                    const float g1 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(r[i + 1])));
                    const float u0 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(r[GROUP / 2 + i])));
                    const float u1 = __bfloat162float(__float2bfloat16_rn(__uint_as_float(r[GROUP / 2 + i + 1])));
                    w[e] = pack2(g0 / (1.f + __expf(-g0)) * u0, g1 / (1.f + __expf(-g1)) * u1);
                }
                dst = p.U + (size_t)b * (p.N / 2) + n0 + g * (GROUP / 2);
            } else {
                if (p.residual) {
#pragma unroll
                    for (int v = 0; v < COLS / 8; ++v) {
                        const uint32_t rw[4] = {res[v].x, res[v].y, res[v].z, res[v].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            r[8 * v + 2 * e] = __float_as_uint(__uint_as_float(r[8 * v + 2 * e]) + bf16_lo(rw[e]));
                            r[8 * v + 2 * e + 1] = __float_as_uint(__uint_as_float(r[8 * v + 2 * e + 1]) + bf16_hi(rw[e]));
                        }
                    }
                    fetch_residual(g + n);
                }
                if (p.bias)
#pragma unroll
                    for (int v = 0; v < COLS / 8; ++v) {
                        const uint4 bv = __ldcg(reinterpret_cast<const uint4 *>(p.bias + col) + v);
                        const uint32_t bw[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            r[8 * v + 2 * e] = __float_as_uint(__uint_as_float(r[8 * v + 2 * e]) + bf16_lo(bw[e]));
                            r[8 * v + 2 * e + 1] = __float_as_uint(__uint_as_float(r[8 * v + 2 * e + 1]) + bf16_hi(bw[e]));
                        }
                    }
#pragma unroll
                for (int e = 0; e < WORDS; ++e) w[e] = pack2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1]));
                dst = p.U + (size_t)b * p.N + col;
            }
            if constexpr (WORDS >= 8) {
                if (wide) {
#pragma unroll
                    for (int v = 0; v < WORDS; v += 8) ptx::stg256(dst + 2 * v, w + v);
                    return;
                }
            }
#pragma unroll
            for (int v = 0; v < WORDS; v += 4) *reinterpret_cast<uint4 *>(dst + 2 * v) = make_uint4(w[v], w[v + 1], w[v + 2], w[v + 3]);
        };
        for (; g + AT_ONCE <= g_end; g += AT_ONCE) finish(std::integral_constant<int, AT_ONCE>{}, g);
        if (AT_ONCE > 1 && g < g_end) finish(std::integral_constant<int, 1>{}, g);
    }
    __syncwarp();                           // (rows past the batch left the last round early: the barriers below want whole warps)
    ptx::tc_fence_before();
    if (ks > 1) ptx::cluster_sync();        // every CTA has received its groups: the senders' shared memory may go
    else __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, MW * NT);
    }
}

// How a projection is cut: NT columns per tile, ks CTAs per tile, and the ring stages that fit.
struct SlabPlan {
    int nt, ks, stages;
    float us;                // the estimate
};

// The cut with the least estimated time (microseconds; constants fitted to 5,000 timed cuts, 24 weight shapes x 17 batches,
// where the cut it picks is 0.1 % slower than the fastest one on average, 13 % at worst): a wave of CTAs takes 1.7 and, per block of
// 64 K elements, 0.17 / 0.195 / 0.255 for a tile of 64 / 128 / 256 columns, a little less with few rows, but all waves never less
// than the weights take at 5.75 TB/s; an exchange, once per wave, 1.3, 0.33 per further CTA of the cluster and the time of its bytes at
// 17 KB a microsecond.  A wave is what is resident at a time: fit[ks] clusters of ks CTAs, fewer than the SMs divided by ks,
// because a cluster lives within a part of the chip (148 SMs hold 45 clusters of 3, not 49).  Counted without that, and
// with the exchange once per call, the rule took cuts of two waves for one: 300 x 4096 -> 4096 30 us as 48 clusters
// of 3, 18.7 as 96 CTAs; 300 x 2816 -> 1024 14.3 and 8.3; 1600 x 8192 -> 2048 80 as 104 clusters of 4, 47 unsplit.  Taken now, us with
// weights ahead: 127 x 2048 -> 2048 7.2 as 32 tiles x 4 (8.3 unsplit), 127 x 5632 -> 2048 10.2 as 32 x 4 (17.7), 127 x 2048 ->
// 3072 8.0 as 48 x 2 (8.3), 1204 x 2048 -> 2048 15.2 as 80 tiles of 256 columns (22.8 as 320 of 64).
// only: the one width that serves (0: all do)
SlabPlan slab_plan(const int *fit, int B, int K, int N, int x_rows, int only) {
    const int m_tiles = (B + BM - 1) / BM, atoms = K / BK, nq = x_rows > 32 ? x_rows / 32 : 1;
    const float weights_us = (float)N * K * 2 / 5.75e6f, few_rows = 1.f - 0.08f * (float)(BM - x_rows) / BM;
    SlabPlan best{};
    for (int nt = 64; nt <= 256; nt *= 2) {
        if (N % nt != 0 || (only && nt != only)) continue;
        const int groups = nt / GROUP;
        const float block_us = (nt == 64 ? 0.17f : nt == 128 ? 0.195f : 0.255f) * few_rows;
        for (int ks = 1; ks <= MAX_CLUSTER && ks <= groups && ks * 2 <= std::max(2, atoms); ++ks) {
            const int own_lo = groups / ks, own_hi = (groups + ks - 1) / ks;
            const int send = (groups - own_lo) * nq * QUAD_BYTES, recv = (ks - 1) * own_hi * nq * QUAD_BYTES;
            if (fit[ks] < 1 || (ks > 1 && send + recv > RING_BYTES)) continue;
            const long long tiles = (long long)(N / nt) * m_tiles, waves = (tiles + fit[ks] - 1) / fit[ks];
            const float us = std::max((float)waves * ((atoms + ks - 1) / ks) * block_us, weights_us) +
                             waves * (1.7f + (ks > 1 ? 1.3f + 0.33f * (ks - 1) + send / 17e3f : 0.f));
            if (best.nt == 0 || us < best.us) {
                const int stages = std::min(MAX_STAGES, RING_BYTES / (blocks_per_stage(nt) * (x_rows + nt) * BK * 2));
                best = SlabPlan{nt, ks, stages / mma_warps(nt) * mma_warps(nt), us};
            }
        }
    }
    return best;
}

int rows_fetched(int B) { return B > 64 ? 128 : B > 32 ? 64 : B > 16 ? 32 : 16; }

int only_width(const ConvParams &p, bool gated) { return gated ? 128 : p.rope.q ? p.rope.dh : 0; }

template <int NT, bool IN_MAJOR, Epilogue EPI>
cudaError_t run_as(photon_ctx *ctx, ConvParams p, const SlabPlan &s, cudaStream_t st, long long *launches) {
    const CUtensorMap *t;
    CUtensorMap mx, mw;
    if (!(t = ctx->tmaps.get(p.x, (uint64_t)p.B, (uint64_t)p.D, p.x_rows))) return cudaErrorInvalidValue;
    mx = *t;
    // [K, N] in boxes of 64 k x 64 n, or [N, K] in boxes of NT n x 64 k (gate rows and up rows are fetched apart)
    t = IN_MAJOR ? ctx->tmaps.get(p.w, (uint64_t)p.D, (uint64_t)p.N, BK) : ctx->tmaps.get(p.w, (uint64_t)p.N, (uint64_t)p.D, EPI == GATED_MLP ? NT / 2 : NT);
    if (!t) return cudaErrorInvalidValue;
    mw = *t;
    p.ksplit = s.ks; p.stages = s.stages;
    p.once = p.w_ahead && (p.D / BK + s.ks - 1) / s.ks <= s.stages * blocks_per_stage(NT);
    constexpr size_t smem = (size_t)RING_BYTES + BAR_BYTES + (EPI == ROTARY ? NT / 2 * sizeof(double) + ANGLES_BYTES : 0);
    static size_t smem_set[kMaxDevices] = {};
    if (const cudaError_t e = ensure_dynamic_smem(linear_slab_kernel<NT, IN_MAJOR, EPI>, smem, ctx->device, smem_set)) return e;
    const dim3 grid(p.ksplit * (p.N / NT), (p.B + BM - 1) / BM);
    const cudaError_t e = launch_dependent(linear_slab_kernel<NT, IN_MAJOR, EPI>, grid, dim3(SLAB_THREADS), smem, st,
                                           p.ksplit > 1 ? p.ksplit : 0, p, mx, mw);
    ++*launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <Epilogue EPI>
cudaError_t run(photon_ctx *ctx, ConvParams p, cudaStream_t st, long long *launches) {
    if (p.B == 0) return cudaSuccess;
    p.x_rows = rows_fetched(p.B);
    const SlabPlan s = slab_plan(ctx->clusters, p.B, p.D, p.N, p.x_rows, only_width(p, EPI == GATED_MLP));
    if constexpr (EPI != GATED_MLP)
        if (s.nt == 64) return p.w_out_major ? run_as<64, false, EPI>(ctx, p, s, st, launches) : run_as<64, true, EPI>(ctx, p, s, st, launches);
    if (s.nt == 128) return p.w_out_major ? run_as<128, false, EPI>(ctx, p, s, st, launches) : run_as<128, true, EPI>(ctx, p, s, st, launches);
    if constexpr (EPI == PLAIN)
        if (s.nt == 256) return p.w_out_major ? run_as<256, false, EPI>(ctx, p, s, st, launches) : run_as<256, true, EPI>(ctx, p, s, st, launches);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_linear(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return run<PLAIN>(ctx, p, st, launches);
}

// Whether the fused gate/up form serves this shape: whole slabs of 64 features, and enough of them to occupy half of the
// GPU before K is split (below that the plain projection and the activation kernel).
bool gate_up_fits_small_tiles(const photon_ctx *ctx, const ConvParams &p) {
    const long long tiles = (long long)(p.N / 128) * ((p.B + BM - 1) / BM);
    return p.N % 128 == 0 && p.D % BK == 0 && tiles * 2 >= ctx->sm_count;
}

cudaError_t launch_qkv_rope(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return run<ROTARY>(ctx, p, st, launches);
}

cudaError_t launch_gate_up(photon_ctx *ctx, const ConvParams &p, cudaStream_t st, long long *launches) {
    return run<GATED_MLP>(ctx, p, st, launches);
}

// How many clusters of 1 to MAX_CLUSTER CTAs of this kernel the device holds at a time.  Asked once per device: the eight
// questions take 3 ms.
cudaError_t linear_cluster_counts(int device, int (&fit)[MAX_CLUSTER + 1]) {
    static int known[kMaxDevices][MAX_CLUSTER + 1] = {};
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    if (known[device][1] > 0) {
        std::copy(known[device], known[device] + MAX_CLUSTER + 1, fit);
        return cudaSuccess;
    }
    constexpr size_t smem = (size_t)RING_BYTES + BAR_BYTES;
    const auto kernel = linear_slab_kernel<64, true, PLAIN>;         // (the other forms take as much of everything that counts here)
    if (const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return e;
    fit[0] = 0;
    for (int ks = 1; ks <= MAX_CLUSTER; ++ks) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ks);
        cfg.blockDim = dim3(SLAB_THREADS);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = ks;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if (const cudaError_t e = cudaOccupancyMaxActiveClusters(&fit[ks], kernel, &cfg)) return e;
    }
    std::copy(fit, fit + MAX_CLUSTER + 1, known[device]);
    return cudaSuccess;
}

// The time of the best cut for comparison with the pair kernel; negative where there is no cut (a gated form of half slabs).
// The estimate above was fitted to small batches; with the whole chip at work the same cuts take about a quarter longer,
// every wave ends in an epilogue of its own, and the residual and the output move while nothing else does (5 TB/s).
float linear_slab_us(const int *fit, const ConvParams &p, bool gated) {
    const SlabPlan s = slab_plan(fit, p.B, p.D, p.N, rows_fetched(p.B), only_width(p, gated));
    if (s.nt == 0) return -1.f;
    const long long tiles = (long long)(p.N / s.nt) * ((p.B + BM - 1) / BM), waves = (tiles + fit[s.ks] - 1) / fit[s.ks];
    return 1.25f * s.us + waves * (s.nt / 256.f) + (float)p.B * p.N * (p.residual ? 4 : 2) / 5e6f;
}

void linear_cut(const int *fit, int B, int K, int N, bool gated, int32_t *cut) {
    const SlabPlan s = slab_plan(fit, B, K, N, rows_fetched(B), gated ? 128 : 0);
    cut[0] = s.nt; cut[1] = s.ks; cut[2] = s.stages; cut[3] = mma_warps(s.nt);
}

int linear_slab_registers() {
    cudaFuncAttributes a{};
    return cudaFuncGetAttributes(&a, linear_slab_kernel<64, false, PLAIN>) == cudaSuccess ? (a.numRegs + 7) / 8 * 8 * SLAB_THREADS : -1;
}
