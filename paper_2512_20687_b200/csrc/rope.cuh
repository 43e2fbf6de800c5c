// Rotary encoding: the angles, and the epilogue of a fused q/k/v projection that rotates, splits and appends (see RopeOut).
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace rope {

// The inverse wavelength of feature pair j.
__device__ __forceinline__ double inverse_wavelength(int j, int dh, double log2_theta) { return exp2(-2.0 * (double)j / dh * log2_theta); }

// Cosine and sine at a position: the angle and its reduction to [-pi, pi] in double precision (positions reach thousands of radians,
// which single-precision sines do not survive), sine and cosine of the remainder in single.
__device__ __forceinline__ void angle(int at, double inv, float *c, float *s) {
    const double a = (double)at * inv;
    const double turns = rint(a * 0.15915494309189535);
    __sincosf((float)fma(turns, -6.283185307179586, a), s, c);
}

// Cosines and sines of the positions [0, rows) in shared memory; others are computed.  (An SM computes about one angle a clock, for the
// double-precision part of it: 128 rows x 64 features took 4 us, as long as a tile's MMAs at K = 1024, and the projection of 16384
// chunks 112 instead of 75 us.)
struct Table {
    float2 *t;               // [rows][stride]
    const double *inv;       // [dh / 2]
    int rows, half, stride;
    __device__ __forceinline__ void fill(int tid, int threads) {
        for (int i = tid; i < rows * half; i += threads) {
            float2 cs;
            angle(i / half, inv[i % half], &cs.x, &cs.y);
            t[i / half * stride + i % half] = cs;
        }
    }
    template <int N>
    __device__ __forceinline__ void get(int at, int j, float (&c)[N], float (&s)[N]) const {
        if ((unsigned)at < (unsigned)rows) {
            const float2 *row = t + at * stride + j;
#pragma unroll
            for (int e = 0; e < N; ++e) { c[e] = row[e].x; s[e] = row[e].y; }
        } else {
#pragma unroll 1
            for (int e = 0; e < N; ++e) {
                float ce, se;
                angle(at, inv[j + e], &ce, &se);
#pragma unroll
                for (int i = 0; i < N; ++i) if (i == e) { c[i] = ce; s[i] = se; }
            }
        }
    }
};
// Positions that a projection of p has: those below its period, or below the capacity.
__host__ __device__ inline int positions(const RopeOut &r) { return r.period ? r.period : r.cap; }
__host__ __device__ inline int table_stride(int dh) { return dh / 2 + 1; }           // (rows a bank apart)

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&t);
}

// Where row b of the projection goes.
struct Row {
    int b, at;               // row; position
    long long cache;         // cache row of KV head 0 (the next head's is `cap` further on), negative: none
    __device__ __forceinline__ Row() : b(0), at(0), cache(-1) {}
    __device__ __forceinline__ Row(const RopeOut &r, int row) : b(row), at(0), cache(-1) {
        if (r.period) {
            const int i = b / r.period, t = b % r.period, u = r.unit_ids ? __ldcg(r.unit_ids + i) : i;
            at = t;
            if (u < 0 || u >= r.n_units) return;
            const int n = __ldcg(r.len + u);
            if (n >= 0 && n + r.period <= r.cap) cache = (long long)u * r.Hkv * r.cap + n + t;
        } else {
            at = __ldcg(r.len + b);
            if (at >= 0 && at < r.cap) cache = (long long)b * r.Hkv * r.cap + at;
        }
    }
};

// N features [j, j + N) of head h and their partners dh / 2 further on, as they leave the accumulator (fp32 bits): rounded to bf16
// as the projection's output is, rotated (c, s: N cosines and sines) or copied, stored.  N is 8 or 16: whole sectors with 16 (the
// projection of 16384 chunks 119 -> 112 us, before the table).
template <int N>
__device__ __forceinline__ void store(const RopeOut &r, const Row &row, int h, int j, const uint32_t *lo, const uint32_t *hi, const float *c,
                                      const float *s) {
    uint32_t wl[N / 2], wh[N / 2];
    auto put = [&](bf16 *dst) {
        if constexpr (N == 16) {                                // whole sectors
            if ((reinterpret_cast<uintptr_t>(dst) & 31u) == 0) {
                ptx::stg256(dst, wl);
                ptx::stg256(dst + r.dh / 2, wh);
                return;
            }
        }
#pragma unroll
        for (int v = 0; v < N / 8; ++v) {
            *reinterpret_cast<uint4 *>(dst + 8 * v) = make_uint4(wl[4 * v], wl[4 * v + 1], wl[4 * v + 2], wl[4 * v + 3]);
            *reinterpret_cast<uint4 *>(dst + r.dh / 2 + 8 * v) = make_uint4(wh[4 * v], wh[4 * v + 1], wh[4 * v + 2], wh[4 * v + 3]);
        }
    };
#pragma unroll
    for (int e = 0; e < N / 2; ++e) {
        wl[e] = pack2(__uint_as_float(lo[2 * e]), __uint_as_float(lo[2 * e + 1]));
        wh[e] = pack2(__uint_as_float(hi[2 * e]), __uint_as_float(hi[2 * e + 1]));
    }
    if (r.qkv) put(r.qkv + ((size_t)row.b * (r.Hq + 2 * r.Hkv) + h) * r.dh + j);
    const int kv = h - r.Hq;                                    // 0 .. Hkv - 1: a key head, Hkv .. : a value head
    if (kv < r.Hkv) {
#pragma unroll
        for (int e = 0; e < N / 2; ++e) {
            const float a0 = bf16_lo(wl[e]), a1 = bf16_hi(wl[e]), b0 = bf16_lo(wh[e]), b1 = bf16_hi(wh[e]);
            wl[e] = pack2(a0 * c[2 * e] - b0 * s[2 * e], a1 * c[2 * e + 1] - b1 * s[2 * e + 1]);
            wh[e] = pack2(b0 * c[2 * e] + a0 * s[2 * e], b1 * c[2 * e + 1] + a1 * s[2 * e + 1]);
        }
        if (kv < 0) { put(r.q + ((size_t)row.b * r.Hq + h) * r.dh + j); return; }
    }
    const int head = kv < r.Hkv ? kv : kv - r.Hkv;
    bf16 *copy = kv < r.Hkv ? r.k_new : r.v_new;
    if (copy) put(copy + ((size_t)row.b * r.Hkv + head) * r.dh + j);
    if (row.cache >= 0) put((kv < r.Hkv ? r.k_cache : r.v_cache) + (row.cache + (long long)head * r.cap) * r.dh + j);
}

}  // namespace rope
