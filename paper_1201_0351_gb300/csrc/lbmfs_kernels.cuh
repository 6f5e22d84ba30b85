// Device code of the free-surface LBM step (Bogner & Ruede, Sec. 2), templated
// on the population storage.  Included by one translation unit per storage:
//   S = 0  f_q as double, double arithmetic.  Every operation is written in the
//          same order as the plain CPU restatement of the method and the unit is
//          compiled with -fmad=false, so this path reproduces it bit for bit
//          (except for the order of the parallel force / ledger sums);
//   S = 1  f_q - w_q as float, float arithmetic on deviations;
//   S = 2  f_q - w_q as half (q >= 1, times 2^10) with a float rest population
//          chosen so that the stored cell sum equals the collision density.
// Interface mass, fill level, forces, torques and the ledger are double in all
// three.
#pragma once
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lbmfs_internal.h"

namespace lbmfs {
namespace {  // internal linkage: one copy per storage translation unit

// ----------------------------------------------------------------- lattice
// D3Q19 in the order C,W,E,N,S,T,B,TW,TE,TN,TS,NW,NE,SW,SE,BW,BE,BN,BS (the
// order of the paper's stencil figure, Eq. links).
__host__ __device__ __forceinline__ constexpr int cx(int q) {
    return q == 1 || q == 7 || q == 11 || q == 13 || q == 15 ? -1
           : (q == 2 || q == 8 || q == 12 || q == 14 || q == 16 ? 1 : 0);
}
__host__ __device__ __forceinline__ constexpr int cy(int q) {
    return q == 3 || q == 9 || q == 11 || q == 12 || q == 17 ? 1
           : (q == 4 || q == 10 || q == 13 || q == 14 || q == 18 ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int cz(int q) {
    return q == 5 || (q >= 7 && q <= 10) ? 1 : (q == 6 || q >= 15 ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int opp(int q) {
    // C-C, W-E, N-S, T-B, TW-BE, TE-BW, TN-BS, TS-BN, NW-SE, NE-SW
    return q == 0 ? 0
                  : (q <= 6 ? (q & 1 ? q + 1 : q - 1)
                            : (q == 7 || q == 8 || q == 15 || q == 16 ? 23 - q
                                                                      : (q <= 14 && q >= 11 ? 25 - q : 27 - q)));
}
// the table is checked at compile time: c_opp(q) = -c_q, weights symmetric
__host__ __device__ constexpr bool lattice_ok() {
    for (int q = 0; q < 19; ++q) {
        int p = opp(q);
        if (cx(p) != -cx(q) || cy(p) != -cy(q) || cz(p) != -cz(q)) return false;
        int s = (cx(q) != 0) + (cy(q) != 0) + (cz(q) != 0);
        if ((q == 0) != (s == 0) || (q >= 1 && q <= 6) != (s == 1) || (q >= 7) != (s == 2)) return false;
    }
    return true;
}
static_assert(lattice_ok(), "D3Q19 table");
// weights of the stencil figure caption: 1/3, 1/18, 1/36
__host__ __device__ __forceinline__ constexpr double wd(int q) {
    return q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
}
__host__ __device__ __forceinline__ constexpr float wf(int q) {
    return q == 0 ? 1.0f / 3.0f : (q <= 6 ? 1.0f / 18.0f : 1.0f / 36.0f);
}

#ifndef LBMFS_BULK_MINB
#define LBMFS_BULK_MINB 8  // resident blocks per SM asked of ptxas for the bulk kernel (64 registers)
#endif
#ifndef LBMFS_BULK_ZB
#define LBMFS_BULK_ZB 8    // z-planes per block of the TMA-staged bulk kernel (those of the default kernel: bulk_planes)
#endif
#ifndef LBMFS_BULK_PIPE_ZB
#define LBMFS_BULK_PIPE_ZB 16  // z-planes per block of the software-pipelined bulk kernel
#endif
#ifndef LBMFS_FORCE_MINB
#define LBMFS_FORCE_MINB 6  // resident 128-thread blocks per SM of the float-storage force kernel (80 registers)
#endif
#ifndef LBMFS_IFACE_MINB
#define LBMFS_IFACE_MINB 6  // resident blocks per SM asked of ptxas for the interface kernel (80 registers)
#endif
#ifndef LBMFS_IFACE_GRID
#define LBMFS_IFACE_GRID (16 * 152)  // blocks of the single-tank interface kernel (16 per SM)
#endif
#ifndef LBMFS_ST_CS
#define LBMFS_ST_CS 0      // population stores with the evict-first (streaming) hint
#endif
constexpr float F16_SCALE = 1024.0f;
constexpr float F16_INV_SCALE = 1.0f / 1024.0f;
constexpr int CL_WALL = 256;

// ----------------------------------------------------------------- storage
// population loads / stores (tuning knob: evict-first stores)
template <class T> __device__ __forceinline__ T pop_ld(const T *p) { return *p; }
// through the read-only data path: only for a grid that no thread of the
// launch writes (the bulk kernel's source populations)
template <class T> __device__ __forceinline__ T pop_ldg(const T *p) { return __ldg(p); }
template <class T> __device__ __forceinline__ void pop_st(T *p, T v) {
#if LBMFS_ST_CS
    __stcs(p, v);
#else
    *p = v;
#endif
}
template <int S> struct Sto;

template <> struct Sto<0> {
    using R = double;
    static constexpr bool shifted = false;
    static __device__ __forceinline__ double ld(const void *g, int q, long long i, long long N) {
        return pop_ld(reinterpret_cast<const double *>(g) + ((long long)q * N + i));
    }
    static __device__ __forceinline__ double ldg(const void *g, int q, long long i, long long N) {
        return pop_ldg(reinterpret_cast<const double *>(g) + ((long long)q * N + i));
    }
    static __device__ __forceinline__ void st(void *g, int q, long long i, long long N, double v) {
        pop_st(reinterpret_cast<double *>(g) + ((long long)q * N + i), v);
    }
    // value of f_q as double
    static __device__ __forceinline__ double ldf(const void *g, int q, long long i, long long N) {
        return ld(g, q, i, N);
    }
    // store a full cell given as 19 doubles f_q
    static __device__ __forceinline__ void st_cell(void *g, long long i, long long N, const double *f) {
#pragma unroll
        for (int q = 0; q < Q; ++q) st(g, q, i, N, f[q]);
    }
    static size_t bytes(long long N) { return (size_t)N * Q * sizeof(double); }
    static constexpr int SCALE = 1;
    static __device__ __forceinline__ double ld_raw(const void *g, int q, long long i, long long N) { return ld(g, q, i, N); }
    static __device__ __forceinline__ double ldg_raw(const void *g, int q, long long i, long long N) {
        return ldg(g, q, i, N);
    }
};

template <> struct Sto<1> {
    using R = float;
    static constexpr bool shifted = true;
    static __device__ __forceinline__ float ld(const void *g, int q, long long i, long long N) {
        return pop_ld(reinterpret_cast<const float *>(g) + ((long long)q * N + i));
    }
    static __device__ __forceinline__ float ldg(const void *g, int q, long long i, long long N) {
        return pop_ldg(reinterpret_cast<const float *>(g) + ((long long)q * N + i));
    }
    static __device__ __forceinline__ void st(void *g, int q, long long i, long long N, float v) {
        pop_st(reinterpret_cast<float *>(g) + ((long long)q * N + i), v);
    }
    static __device__ __forceinline__ double ldf(const void *g, int q, long long i, long long N) {
        return wd(q) + (double)ld(g, q, i, N);
    }
    static __device__ __forceinline__ void st_cell(void *g, long long i, long long N, const double *f) {
#pragma unroll
        for (int q = 0; q < Q; ++q) st(g, q, i, N, (float)(f[q] - wd(q)));
    }
    // store the collided deviations dv; the rest population is replaced by
    // dp_0 + sum_{q>=1} (dp_q - dv_q) (equal to dv_0 in exact arithmetic) so
    // that the stored cell sum equals the streamed-in sum of dp up to one
    // rounding of a small number: no mass drift from float rounding
    static __device__ __forceinline__ void st_dev(void *g, long long i, long long N, const float *dv, const float *dp) {
        float rest = 0.0f;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            st(g, q, i, N, dv[q]);
            rest += dp[q] - dv[q];
        }
        st(g, 0, i, N, dp[0] + rest);
    }
    static size_t bytes(long long N) { return (size_t)N * Q * sizeof(float); }
    // store one deviation, return the value as stored
    static __device__ __forceinline__ float st_one(void *g, int q, long long i, long long N, float v) {
        st(g, q, i, N, v);
        return v;
    }
    // values as stored (no scale)
    static constexpr int SCALE = 1;
    static __device__ __forceinline__ float ld_raw(const void *g, int q, long long i, long long N) { return ld(g, q, i, N); }
    static __device__ __forceinline__ float ldg_raw(const void *g, int q, long long i, long long N) { return ldg(g, q, i, N); }
    static __device__ __forceinline__ float st_raw(void *g, int q, long long i, long long N, float v) {
        return st_one(g, q, i, N, v);
    }
};

template <> struct Sto<2> {
    using R = float;
    static constexpr bool shifted = true;
    // plane 0: float (N); planes 1..18: half (N each), after it
    static __device__ __forceinline__ const __half *hp(const void *g, long long N) {
        return reinterpret_cast<const __half *>(reinterpret_cast<const float *>(g) + N);
    }
    static __device__ __forceinline__ float ld(const void *g, int q, long long i, long long N) {
        if (q == 0) return pop_ld(reinterpret_cast<const float *>(g) + i);
        return __half2float(pop_ld(hp(g, N) + ((long long)(q - 1) * N + i))) * F16_INV_SCALE;
    }
    static __device__ __forceinline__ float ldg(const void *g, int q, long long i, long long N) {
        if (q == 0) return pop_ldg(reinterpret_cast<const float *>(g) + i);
        return __half2float(pop_ldg(hp(g, N) + ((long long)(q - 1) * N + i))) * F16_INV_SCALE;
    }
    static __device__ __forceinline__ double ldf(const void *g, int q, long long i, long long N) {
        return wd(q) + (double)ld(g, q, i, N);
    }
    // d*_q for q >= 1 rounded to half; the rest population takes
    // dp_0 + sum_{q>=1} (dp_q - dequant(h_q)) so that the stored cell sum
    // equals the streamed-in sum of dp (the collision density) up to one
    // rounding of a small number
    static __device__ __forceinline__ void st_dev(void *g, long long i, long long N, const float *dv, const float *dp) {
        __half *h = const_cast<__half *>(hp(g, N));
        float rest = 0.0f;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            __half hq = __float2half_rn(dv[q] * F16_SCALE);
            pop_st(h + ((long long)(q - 1) * N + i), hq);
            rest += dp[q] - __half2float(hq) * F16_INV_SCALE;
        }
        pop_st(reinterpret_cast<float *>(g) + i, dp[0] + rest);
    }
    static __device__ __forceinline__ void st_cell(void *g, long long i, long long N, const double *f) {
        float dv[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) dv[q] = (float)(f[q] - wd(q));
        st_dev(g, i, N, dv, dv);
    }
    static size_t bytes(long long N) { return (size_t)N * (sizeof(float) + (Q - 1) * sizeof(__half)); }
    static __device__ __forceinline__ float st_one(void *g, int q, long long i, long long N, float v) {
        if (q == 0) {
            pop_st(reinterpret_cast<float *>(g) + i, v);
            return v;
        }
        __half hq = __float2half_rn(v * F16_SCALE);
        pop_st(const_cast<__half *>(hp(g, N)) + ((long long)(q - 1) * N + i), hq);
        return __half2float(hq) * F16_INV_SCALE;
    }
    // values as stored: q >= 1 times F16_SCALE, the rest population unscaled
    static constexpr int SCALE = (int)F16_SCALE;
    static __device__ __forceinline__ float ld_raw(const void *g, int q, long long i, long long N) {
        if (q == 0) return pop_ld(reinterpret_cast<const float *>(g) + i);
        return __half2float(pop_ld(hp(g, N) + ((long long)(q - 1) * N + i)));
    }
    static __device__ __forceinline__ float ldg_raw(const void *g, int q, long long i, long long N) {
        if (q == 0) return pop_ldg(reinterpret_cast<const float *>(g) + i);
        return __half2float(pop_ldg(hp(g, N) + ((long long)(q - 1) * N + i)));
    }
    static __device__ __forceinline__ float st_raw(void *g, int q, long long i, long long N, float v) {
        if (q == 0) {
            pop_st(reinterpret_cast<float *>(g) + i, v);
            return v;
        }
        __half hq = __float2half_rn(v);
        pop_st(const_cast<__half *>(hp(g, N)) + ((long long)(q - 1) * N + i), hq);
        return __half2float(hq);
    }
};

// ---------------------------------------------------------------- helpers

// Programmatic launch: lets a kernel that was launched as this one's dependent
// begin once all of this launch's blocks have got here.  The bulk kernel is
// launched so behind the force kernel, which it does not depend on: the force
// kernel's few blocks, the first of a chain of short kernels, then get their
// SMs before the bulk kernel's blocks fill the GPU.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// In a kernel so launched that does depend on the one before it: waits for that
// one's end (nothing to wait for otherwise).  The launch itself is then already
// behind it, about 1.5 us of each short kernel in a chain.
__device__ __forceinline__ void wait_for_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
// order earlier generic-proxy accesses to shared memory before the async-proxy
// (bulk copy) writes that follow
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ long long nbr(const Dev &d, int x, int y, int z, int dx, int dy, int dz) {
    int px = x + dx, py = y + dy, pz = z + dz;
    if (px < 0 || px >= d.nx) {
        if (!(d.periodic & 1u)) return -1;
        px = px < 0 ? px + d.nx : px - d.nx;
    }
    if (py < 0 || py >= d.ny) {
        if (!(d.periodic & 2u)) return -1;
        py = py < 0 ? py + d.ny : py - d.ny;
    }
    if (pz < 0 || pz >= d.nz) {
        if (!(d.periodic & 4u)) return -1;
        pz = pz < 0 ? pz + d.nz : pz - d.nz;
    }
    return px + (long long)d.nx * (py + (long long)d.ny * pz);
}

__device__ __forceinline__ void coords(const Dev &d, long long idx, int &x, int &y, int &z) {
    // every cell index is below 2^32 (checked at create): 32-bit divisions
    const uint32_t i = (uint32_t)idx, r = i / (uint32_t)d.nx;
    x = (int)(i - r * (uint32_t)d.nx);
    z = (int)(r / (uint32_t)d.ny);
    y = (int)(r - (uint32_t)z * (uint32_t)d.ny);
}

// class of cell i (the flag byte without the neighbour-obstacle bit); walls
// (i < 0) report CL_WALL
__device__ __forceinline__ int clsv(const Dev &d, long long i) { return (int)(d.flags[i] & CL_MASK); }
__device__ __forceinline__ int cls(const Dev &d, long long i) { return i < 0 ? CL_WALL : clsv(d, i); }
__device__ __forceinline__ void set_cls(const Dev &d, long long i, int c) {
    d.flags[i] = (uint8_t)((d.flags[i] & ~CL_MASK) | c);
}

// warp-aggregated append of val to a worklist
__device__ __forceinline__ void wl_append(const Dev &d, bool pred, int list, uint32_t val) {
    unsigned act = __activemask();
    unsigned mask = __ballot_sync(act, pred);
    if (!pred) return;
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&d.cnt[list], (uint32_t)__popc(mask));
    base = __shfl_sync(mask, base, leader);
    uint32_t pos = base + (uint32_t)__popc(mask & ((1u << lane) - 1u));
    if (pos < d.cap) d.list[list][pos] = val;
    else atomicOr(d.status, ST_OVERFLOW);
}

__device__ __forceinline__ uint32_t wl_count(const Dev &d, int list) {
    uint32_t c = *reinterpret_cast<volatile uint32_t *>(&d.cnt[list]);
    return c < d.cap ? c : d.cap;
}

// components of a direction known at run time only (a lane's), 2 bits each
__host__ __device__ constexpr unsigned long long dir_bits(int axis) {
    unsigned long long b = 0;
    for (int q = 0; q < Q; ++q)
        b |= (unsigned long long)((axis == 0 ? cx(q) : (axis == 1 ? cy(q) : cz(q))) + 1) << (2 * q);
    return b;
}
__device__ __forceinline__ int dir_x(int q) { return (int)((dir_bits(0) >> (2 * q)) & 3u) - 1; }
__device__ __forceinline__ int dir_y(int q) { return (int)((dir_bits(1) >> (2 * q)) & 3u) - 1; }
__device__ __forceinline__ int dir_z(int q) { return (int)((dir_bits(2) >> (2 * q)) & 3u) - 1; }

// The cells that may be interface in this step: the interface cells that the
// previous step's bulk pass met, then those its conversions (from gas, from
// liquid) and its remap may have added, as one sequence.  The sets are
// disjoint (a cell was interface, gas, liquid or obstacle at the start of that
// step); an entry whose class is no longer interface is passed over.  So the
// interface kernel needs no list from this step's bulk pass and runs beside
// it.
struct IfaceSeq {
    uint32_t e[PREV_LISTS];  // ends of the parts
};
__device__ __forceinline__ IfaceSeq iface_seq(const Dev &d) {
    IfaceSeq r;
    uint32_t t = 0;
#pragma unroll
    for (int k = 0; k < PREV_LISTS; ++k) {
        const uint32_t c = d.pcnt[prev_wl(k)];
        t += c < d.cap ? c : d.cap;
        r.e[k] = t;
    }
    return r;
}
__device__ __forceinline__ uint32_t iface_cell(const Dev &d, const IfaceSeq &r, uint32_t it) {
    const uint32_t *p = d.plist[0] + it;
#pragma unroll
    for (int k = 1; k < PREV_LISTS; ++k)
        if (it >= r.e[k - 1]) p = d.plist[k] + (it - r.e[k - 1]);
    return *p;
}

// opposite of a direction known at run time only
__host__ __device__ constexpr unsigned long long opp_bits(int half) {
    unsigned long long b = 0;
    for (int q = 10 * half; q < (half ? Q : 10); ++q) b |= (unsigned long long)opp(q) << (5 * (q - 10 * half));
    return b;
}
__device__ __forceinline__ int opp_lane(int q) {
    return (int)((q < 10 ? opp_bits(0) >> (5 * q) : opp_bits(1) >> (5 * (q - 10))) & 31u);
}

// atomic OR / AND on one byte of the mark array; returns the old byte
__device__ __forceinline__ uint8_t mark_or(const Dev &d, long long i, uint8_t bits) {
    uintptr_t a = reinterpret_cast<uintptr_t>(d.cmark + i);
    unsigned int *w = reinterpret_cast<unsigned int *>(a & ~(uintptr_t)3);
    unsigned sh = (unsigned)(a & 3) * 8u;
    unsigned old = atomicOr(w, (unsigned)bits << sh);
    return (uint8_t)(old >> sh);
}
__device__ __forceinline__ void mark_and(const Dev &d, long long i, uint8_t bits) {
    uintptr_t a = reinterpret_cast<uintptr_t>(d.cmark + i);
    unsigned int *w = reinterpret_cast<unsigned int *>(a & ~(uintptr_t)3);
    unsigned sh = (unsigned)(a & 3) * 8u;
    atomicAnd(w, ~((unsigned)bits << sh));
}

__device__ __forceinline__ double min_image(const Dev &d, double v, int k) {
    if (d.periodic & (1u << k)) {
        double n = k == 0 ? (double)d.nx : (k == 1 ? (double)d.ny : (double)d.nz);
        v = v - n * floor(v / n + 0.5);
    }
    return v;
}

// rotation matrix of the unit quaternion (w, x, y, z), row-major
__device__ __forceinline__ void rotation(const double *q, double *R) {
    double w = q[0], x = q[1], y = q[2], z = q[3];
    R[0] = 1.0 - 2.0 * (y * y + z * z);
    R[1] = 2.0 * (x * y - w * z);
    R[2] = 2.0 * (x * z + w * y);
    R[3] = 2.0 * (x * y + w * z);
    R[4] = 1.0 - 2.0 * (x * x + z * z);
    R[5] = 2.0 * (y * z - w * x);
    R[6] = 2.0 * (x * z - w * y);
    R[7] = 2.0 * (y * z + w * x);
    R[8] = 1.0 - 2.0 * (x * x + y * y);
}

// Sec. 2.3: cell centre strictly inside the body (box, or sphere of radius
// h[0]); products and sums rounded one by one (no fused multiply-add) so that
// every storage classifies a centre on the surface the same way
// Float pre-test of the cell-centre-inside rule: 1 inside, 0 outside, -1
// undecided.  The cell centre relative to the body comes from the integer part
// and the fraction of the centre (exact integer, fraction rounded once), the
// rotation and the extents in float; every decision keeps a margin of
// 1e-5 (1 + |d|_1 + h) to the surface, well above the float evaluation's error
// bound (a few times 2^-24 (1 + |d|_1 + h)), so where it decides the double
// test below gives the same answer.  GB300's double rate is 1/64 of its float
// rate, and most cells of a body's range lie far from its surface.
__device__ __forceinline__ int inside_float(const Body &b, int x, int y, int z) {
    const float df[3] = {(float)(x - b.oi[0]) + (0.5f - b.of[0]), (float)(y - b.oi[1]) + (0.5f - b.of[1]),
                         (float)(z - b.oi[2]) + (0.5f - b.of[2])};
    const float s = fabsf(df[0]) + fabsf(df[1]) + fabsf(df[2]);
    if (b.shape == 1) {
        const float r2 = df[0] * df[0] + df[1] * df[1] + df[2] * df[2];
        const float m = 1e-5f * (1.0f + s + r2 + b.hf[0]);  // hf[0] holds the squared radius
        return r2 < b.hf[0] - m ? 1 : (r2 > b.hf[0] + m ? 0 : -1);
    }
    int res = 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = fabsf(b.Rf[0 * 3 + k] * df[0] + b.Rf[1 * 3 + k] * df[1] + b.Rf[2 * 3 + k] * df[2]);
        const float m = 1e-5f * (1.0f + s + b.hf[k]);
        if (a > b.hf[k] + m) return 0;
        if (!(a < b.hf[k] - m)) res = -1;
    }
    return res;
}
__device__ __forceinline__ bool inside(const Dev &d, const Body &b, int x, int y, int z) {
    if (!d.periodic) {
        const int r = inside_float(b, x, y, z);
        if (r >= 0) return r != 0;
    }
    double dd[3] = {min_image(d, (x + 0.5) - b.o[0], 0), min_image(d, (y + 0.5) - b.o[1], 1),
                    min_image(d, (z + 0.5) - b.o[2], 2)};
    if (b.shape == 1)
        return __dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])), __dmul_rn(dd[2], dd[2])) <
               __dmul_rn(b.h[0], b.h[0]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double bk = __dadd_rn(__dadd_rn(__dmul_rn(b.R[0 * 3 + k], dd[0]), __dmul_rn(b.R[1 * 3 + k], dd[1])),
                              __dmul_rn(b.R[2 * 3 + k], dd[2]));
        if (!(fabs(bk) < b.h[k])) return false;
    }
    return true;
}

// Eq. noslip at a domain wall: c_q . u_w with u_w the velocity of the face
// that the link (x, q) crosses (source beyond the grid); a link across an edge
// takes the face of its lowest axis
__device__ __forceinline__ int wall_face(const Dev &d, int x, int y, int z, int q) {
    const int p[3] = {x - cx(q), y - cy(q), z - cz(q)}, nn[3] = {d.nx, d.ny, d.nz};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (d.periodic & (1u << k)) continue;
        if (p[k] < 0) return 2 * k;
        if (p[k] >= nn[k]) return 2 * k + 1;
    }
    return -1;
}
__device__ __forceinline__ double wall_cuw(const Dev &d, int x, int y, int z, int q) {
    const int f = wall_face(d, x, y, z, q);
    if (f < 0) return 0.0;
    const double *u = d.wallv + 3 * f;
    return (cx(q) * u[0] + cy(q) * u[1]) + cz(q) * u[2];
}

__device__ __forceinline__ void body_velocity_at(const Dev &d, const Body &b, const double *p, double *uw) {
    double r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) r[k] = min_image(d, p[k] - b.o[k], k);
    double c0 = b.w[1] * r[2] - b.w[2] * r[1];
    double c1 = b.w[2] * r[0] - b.w[0] * r[2];
    double c2 = b.w[0] * r[1] - b.w[1] * r[0];
    uw[0] = b.v[0] + c0;
    uw[1] = b.v[1] + c1;
    uw[2] = b.v[2] + c2;
}

// (c_x u_0 + c_y u_1) + c_z u_2 without the products by the zeros of c_q
__device__ __forceinline__ double dot_c(int q, const double *u) {
    double s = cx(q) ? cx(q) * u[0] : 0.0;
    if (cy(q)) s = cx(q) ? s + cy(q) * u[1] : cy(q) * u[1];
    if (cz(q)) s = (cx(q) || cy(q)) ? s + cz(q) * u[2] : cz(q) * u[2];
    return s;
}
// c_q . u_w with u_w at the midpoint x_c + c_qbar / 2 of the link (x, q)
__device__ __forceinline__ double link_cuw(const Dev &d, const Body &b, int x, int y, int z, int q) {
    int qb = opp(q);
    double p[3] = {(x + 0.5) + 0.5 * cx(qb), (y + 0.5) + 0.5 * cy(qb), (z + 0.5) + 0.5 * cz(qb)};
    double uw[3];
    body_velocity_at(d, b, p, uw);
    return dot_c(q, uw);
}

// the same in float for the float storages: the body state is rounded once
// (positions relative to the body centre stay well inside float precision).
// BodyF holds what a cell's links share: the cell's offset from the body
// centre, rounded from double, and the body's velocities.
struct BodyF {
    float r0[3], v[3], w[3];
};
__device__ __forceinline__ BodyF body_f(const Body &b, int x, int y, int z) {
    return BodyF{{(float)(x - b.o[0]), (float)(y - b.o[1]), (float)(z - b.o[2])},
                 {(float)b.v[0], (float)b.v[1], (float)b.v[2]},
                 {(float)b.w[0], (float)b.w[1], (float)b.w[2]}};
}
__device__ __forceinline__ float link_cuw_f(const Dev &d, const BodyF &b, int q) {
    const int qb = opp(q);
    float r[3] = {b.r0[0] + (0.5f + 0.5f * cx(qb)), b.r0[1] + (0.5f + 0.5f * cy(qb)), b.r0[2] + (0.5f + 0.5f * cz(qb))};
    const int nn[3] = {d.nx, d.ny, d.nz};
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (d.periodic & (1u << k)) r[k] -= (float)nn[k] * floorf(r[k] / (float)nn[k] + 0.5f);
    const float u0 = b.v[0] + (b.w[1] * r[2] - b.w[2] * r[1]);
    const float u1 = b.v[1] + (b.w[2] * r[0] - b.w[0] * r[2]);
    const float u2 = b.v[2] + (b.w[0] * r[1] - b.w[1] * r[0]);
    return (cx(q) * u0 + cy(q) * u1) + cz(q) * u2;
}
__device__ __forceinline__ float link_cuw_f(const Dev &d, const Body &b, int x, int y, int z, int q) {
    return link_cuw_f(d, body_f(b, x, y, z), q);
}

// ------------------------------------------------- double arithmetic (Sec. 2.1)

// Eq. equilibrium, c_s^2 = 1/3
__device__ __forceinline__ double feq_d(int q, double rho, const double *u) {
    double cu = (cx(q) * u[0] + cy(q) * u[1]) + cz(q) * u[2];
    double usq = (u[0] * u[0] + u[1] * u[1]) + u[2] * u[2];
    double t = ((1.0 + 3.0 * cu) + (4.5 * cu) * cu) - 1.5 * usq;
    return (wd(q) * rho) * t;
}

template <int S>
__device__ __forceinline__ double cell_density(const Dev &d, const void *g, long long i) {
    if constexpr (S != 0) {
        // deviations summed in float, as the collision does
        float dr = 0.0f;
#pragma unroll
        for (int q = 0; q < Q; ++q) dr += Sto<S>::ld(g, q, i, d.N);
        return 1.0 + (double)dr;
    }
    double r = 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) r += Sto<S>::ldf(g, q, i, d.N);
    return r;
}

// density and the velocity of the last collision, sum c f / rho - a
template <int S>
__device__ __forceinline__ double cell_rho_u(const Dev &d, const void *g, long long i, double *u) {
    if constexpr (S != 0) {
        float dr = 0.0f, j0 = 0.0f, j1 = 0.0f, j2 = 0.0f;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float v = Sto<S>::ld(g, q, i, d.N);
            dr += v;
            if (cx(q)) j0 += cx(q) * v;
            if (cy(q)) j1 += cy(q) * v;
            if (cz(q)) j2 += cz(q) * v;
        }
        float r = 1.0f + dr;
        u[0] = (double)(j0 / r - d.a_f[0]);
        u[1] = (double)(j1 / r - d.a_f[1]);
        u[2] = (double)(j2 / r - d.a_f[2]);
        return 1.0 + (double)dr;
    }
    double f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q] = Sto<S>::ldf(g, q, i, d.N);
    double r = 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) r += f[q];
    double j0 = 0.0, j1 = 0.0, j2 = 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        j0 += cx(q) * f[q];
        j1 += cy(q) * f[q];
        j2 += cz(q) * f[q];
    }
    u[0] = j0 / r - d.a[0];
    u[1] = j1 / r - d.a[1];
    u[2] = j2 / r - d.a[2];
    return r;
}

// Double BGK collision of the post-stream cell fp -> fnew (Eq. lbgk with Eq.
// forceterm).  GB300 executes 2 double operations per SM and cycle, so the
// double storage's kernels are bound by their number of double operations, and
// the collision is written with as few as keep the oracle's roundings: each
// result is the oracle's expression
//   rho, j = sums in q order; u = j / rho;
//   t = ((1 + 3 cu) + (4.5 cu) cu) - 1.5 u.u,  fe = (w rho) t,
//   F = (w rho) ((tx + ty) + tz),  tx = (3 (cx - ux) + (9 cu) cx) ax, ...
//   f = (f' - omega (f' - fe)) + F
// without its products by the zeros of c_q (x + 0 y = x) and with every value
// that directions share computed once: c_qbar . u = -(c_q . u) exactly, so the
// pair shares 3 cu, 9 cu and (4.5 cu) cu, and a component with c = 0
// contributes (-3 u) a to every such direction.  ZG (ax = ay = 0, gravity
// along z alone, chosen per launch from the uniform parameters) also drops the
// products by those zero accelerations.  Double operations per
// liquid cell of the bulk kernel (wave tank): 612 before, 329 with this, 310 with
// the stored sum checked by exponents; 96^3 bulk kernel 565, 287 and 270 us, now
// within 4 % of 529 G double operations per second.
// Returns rho.
template <bool ZG> __device__ __forceinline__ double collide_d_t(const Dev &d, const double *fp, double *fnew) {
    double rho = fp[0], j0 = 0.0, j1 = 0.0, j2 = 0.0;
#pragma unroll
    for (int q = 1; q < Q; ++q) rho += fp[q];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        if (cx(q) > 0) j0 += fp[q];
        if (cx(q) < 0) j0 -= fp[q];
        if (cy(q) > 0) j1 += fp[q];
        if (cy(q) < 0) j1 -= fp[q];
        if (cz(q) > 0) j2 += fp[q];
        if (cz(q) < 0) j2 -= fp[q];
    }
    const double u[3] = {j0 / rho, j1 / rho, j2 / rho};
    const double us15 = 1.5 * ((u[0] * u[0] + u[1] * u[1]) + u[2] * u[2]);
    const double om = d.omega;
    // per component: 3 (1 - u), 3 (-1 - u), and the term of a direction with c = 0
    double fpos[3], fneg[3], fzero[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        fzero[k] = (3.0 * -u[k]) * d.a[k];
        fpos[k] = 3.0 * (1.0 - u[k]);
        fneg[k] = 3.0 * (-1.0 - u[k]);
    }
    // weight classes: w rho, and with ZG the force of a direction with c_z = 0
    const double wr0 = wd(0) * rho, wr1 = wd(1) * rho, wr2 = wd(7) * rho;
    {
        const double fe = wr0 * (1.0 - us15);
        const double fq = wr0 * (ZG ? fzero[2] : (fzero[0] + fzero[1]) + fzero[2]);
        fnew[0] = (fp[0] - om * (fp[0] - fe)) + fq;
    }
    const double fz1 = wr1 * fzero[2], fz2 = wr2 * fzero[2];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int qb = opp(q);
        if (qb < q) continue;  // each pair once
        const double wr = q <= 6 ? wr1 : wr2;
        double cu = 0.0;
        bool first = true;
        if (cx(q)) {
            cu = cx(q) > 0 ? u[0] : -u[0];
            first = false;
        }
        if (cy(q)) {
            cu = first ? (cy(q) > 0 ? u[1] : -u[1]) : (cy(q) > 0 ? cu + u[1] : cu - u[1]);
            first = false;
        }
        if (cz(q)) cu = first ? (cz(q) > 0 ? u[2] : -u[2]) : (cz(q) > 0 ? cu + u[2] : cu - u[2]);
        const double c3 = 3.0 * cu, c9 = 9.0 * cu, s = (4.5 * cu) * cu;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = h ? qb : q;
            const double t = ((h ? 1.0 - c3 : 1.0 + c3) + s) - us15;
            const double fe = wr * t;
            // (9 cu_p) c_p,k = (9 cu) c_q,k for both members of the pair
            double f0 = fzero[0], f1 = fzero[1], f2 = fzero[2];
            if (!ZG && cx(p)) f0 = ((cx(p) > 0 ? fpos[0] : fneg[0]) + (cx(q) > 0 ? c9 : -c9)) * d.a[0];
            if (!ZG && cy(p)) f1 = ((cy(p) > 0 ? fpos[1] : fneg[1]) + (cy(q) > 0 ? c9 : -c9)) * d.a[1];
            if (cz(p)) f2 = ((cz(p) > 0 ? fpos[2] : fneg[2]) + (cz(q) > 0 ? c9 : -c9)) * d.a[2];
            double fq;
            if (ZG) fq = cz(p) ? wr * f2 : (q <= 6 ? fz1 : fz2);
            else fq = wr * ((f0 + f1) + f2);
            fnew[p] = (fp[p] - om * (fp[p] - fe)) + fq;
        }
    }
    return rho;
}
__device__ __forceinline__ double collide_d(const Dev &d, const double *fp, double *fnew) {
    if (d.a[0] == 0.0 && d.a[1] == 0.0) return collide_d_t<true>(d, fp, fnew);
    return collide_d_t<false>(d, fp, fnew);
}

// ----------------------------------------- float arithmetic on deviations

// ---- the same collision for one cell (V = float) or two cells at once
// (V = float2, GB300's packed FP32 instructions): every operation is written
// out as one correctly rounded add, multiply or fused multiply-add, so both
// forms round each cell identically and a cell's result does not depend on
// whether it was collided alone or in a pair.
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vrcp(float a) { return __frcp_rn(a); }
#ifndef LBMFS_NO_F32X2
#define LBMFS_NO_F32X2 0  // tuning knob: the pair's arithmetic as two scalar operations
#endif
#if LBMFS_NO_F32X2
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
    return make_float2(__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
#else
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
#endif
__device__ __forceinline__ float2 vrcp(float2 a) { return make_float2(__frcp_rn(a.x), __frcp_rn(a.y)); }
template <class V> __device__ __forceinline__ V vbc(float s);
template <> __device__ __forceinline__ float vbc<float>(float s) { return s; }
template <> __device__ __forceinline__ float2 vbc<float2>(float s) { return make_float2(s, s); }
// a - b as one rounding (b * -1 is exact)
template <class V> __device__ __forceinline__ V vsub(V a, V b) { return vfma(b, vbc<V>(-1.0f), a); }
__device__ __forceinline__ bool vpos_finite(float r) { return r > 0.0f && r < 1e30f; }
__device__ __forceinline__ bool vpos_finite(float2 r) { return vpos_finite(r.x) && vpos_finite(r.y); }

// BGK collision with the Luo force term on deviations dp_q = f'_q - w_q (q >= 1
// times SC, a power of two: the FP16 storage's own scale; dp_0 unscaled),
// fused with the store: store(q, dn) writes the collided deviation and returns
// the value as stored.  The rest population is stored as
// dp_0 + sum_{q>=1} (dp_q - stored_q) / SC: equal to the collided rest
// population in exact arithmetic, it makes the stored cell sum equal the
// streamed-in sum up to one rounding (no mass drift from storage rounding).
// For each pair q, qbar the equilibrium and force terms split as
//   f_eq - w = A +- B,  F = C +- D  with
//   A = w dr + w rho (4.5 (c.u)^2 - 1.5 u.u),  B = 3 w rho c.u,
//   C = w rho (9 (c.u)(c.a) - 3 u.a),          D = 3 w rho c.a,
// (c of the pair's member with the positive leading component) so that
//   dn = (1 - omega) dp + (E +- G),  E = omega A + C,  G = omega B + D.
// Returns the collision density.
// ZG (ax = ay = 0: gravity along z alone) leaves out the products by the zero
// accelerations (x + 0 y = x, so every value is the same): 212 instead of 228
// operations.
template <int SC, bool ZG, class V, class Store>
__device__ __forceinline__ V collide_store_v(const Dev &d, const V *dp, Store store) {
    constexpr float sc = (float)SC, isc = 1.0f / (float)SC;
    V dr = dp[0];
#pragma unroll
    for (int q = 1; q < Q; ++q) dr = vfma(dp[q], vbc<V>(isc), dr);
    V j0 = vbc<V>(0.0f), j1 = vbc<V>(0.0f), j2 = vbc<V>(0.0f);
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        if (cx(q) > 0) j0 = vadd(j0, dp[q]);
        if (cx(q) < 0) j0 = vsub(j0, dp[q]);
        if (cy(q) > 0) j1 = vadd(j1, dp[q]);
        if (cy(q) < 0) j1 = vsub(j1, dp[q]);
        if (cz(q) > 0) j2 = vadd(j2, dp[q]);
        if (cz(q) < 0) j2 = vsub(j2, dp[q]);
    }
    const V rho = vadd(vbc<V>(1.0f), dr);
    const V inv = vmul(vrcp(rho), vbc<V>(isc));
    const V ux = vmul(j0, inv), uy = vmul(j1, inv), uz = vmul(j2, inv);
    const V nusq15 = vmul(vfma(uz, uz, vfma(uy, uy, vmul(ux, ux))), vbc<V>(-1.5f));  // -1.5 u.u
    const float om = d.omega_f, om1 = 1.0f - om;
    const float ax = d.a_f[0], ay = d.a_f[1], az = d.a_f[2];
    const V nua3 = vmul(ZG ? vmul(uz, vbc<V>(az)) : vfma(uz, vbc<V>(az), vfma(uy, vbc<V>(ay), vmul(ux, vbc<V>(ax)))),
                        vbc<V>(-3.0f));
    // per weight class: w dr, w rho, 3 w rho (times SC)
    const V wdr1 = vmul(dr, vbc<V>(wf(1) * sc)), wr1 = vmul(rho, vbc<V>(wf(1) * sc));
    const V wdr2 = vmul(dr, vbc<V>(wf(7) * sc)), wr2 = vmul(rho, vbc<V>(wf(7) * sc));
    const V wr13 = vmul(wr1, vbc<V>(3.0f)), wr23 = vmul(wr2, vbc<V>(3.0f));
    // ZG: C of the directions with c_z = 0, and 3 w rho az of those with c_z = 1
    const V c1 = vmul(wr1, nua3), c2 = vmul(wr2, nua3), d1 = vmul(wr13, vbc<V>(az)), d2 = vmul(wr23, vbc<V>(az));
    V rest = vbc<V>(0.0f);
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int qb = opp(q);
        if (qb < q) continue;  // each pair once
        // p: the member whose leading nonzero velocity component is positive
        const int p = (cx(q) > 0 || (cx(q) == 0 && (cy(q) > 0 || (cy(q) == 0 && cz(q) > 0)))) ? q : qb;
        const bool axis = q <= 6;
        const V wdr = axis ? wdr1 : wdr2, wr = axis ? wr1 : wr2, wr3 = axis ? wr13 : wr23;
        V cu = cx(p) ? ux : (cy(p) ? uy : uz);  // the leading component is +1
        if (cx(p) && cy(p) > 0) cu = vadd(cu, uy);
        if (cx(p) && cy(p) < 0) cu = vsub(cu, uy);
        if ((cx(p) || cy(p)) && cz(p) > 0) cu = vadd(cu, uz);
        if ((cx(p) || cy(p)) && cz(p) < 0) cu = vsub(cu, uz);
        const float ca = (float)cx(p) * ax + (float)cy(p) * ay + (float)cz(p) * az;
        const V A = vfma(wr, vfma(vmul(cu, cu), vbc<V>(4.5f), nusq15), wdr);
        const V C = ZG && cz(p) == 0 ? (axis ? c1 : c2) : vmul(wr, vfma(cu, vbc<V>(9.0f * (ZG ? (float)cz(p) * az : ca)), nua3));
        const V E = vfma(A, vbc<V>(om), C);
        const V wcu = vmul(wr3, cu);
        V G;
        if (!ZG) G = vfma(wcu, vbc<V>(om), vmul(wr3, vbc<V>(ca)));
        else if (cz(p) == 0) G = vmul(wcu, vbc<V>(om));
        else if (cz(p) > 0) G = vfma(wcu, vbc<V>(om), axis ? d1 : d2);
        else G = vfma(wcu, vbc<V>(om), vmul(axis ? d1 : d2, vbc<V>(-1.0f)));
        const V dnp = vfma(dp[p], vbc<V>(om1), vadd(E, G));
        const int m = p == q ? qb : q;
        const V dnm = vfma(dp[m], vbc<V>(om1), vsub(E, G));
        rest = vadd(rest, vsub(dp[p], store(p, dnp)));
        rest = vadd(rest, vsub(dp[m], store(m, dnm)));
    }
    store(0, vfma(rest, vbc<V>(isc), dp[0]));
    return rho;
}

// f_eq(rho_g, u) - w as float deviation
__device__ __forceinline__ float feq_dev_f(int q, float drg, float ux, float uy, float uz) {
    float cu = (float)cx(q) * ux + (float)cy(q) * uy + (float)cz(q) * uz;
    float usq = ux * ux + uy * uy + uz * uz;
    float s = 3.0f * cu + 4.5f * cu * cu - 1.5f * usq;
    return wf(q) * (drg + s + drg * s);
}

// ------------------------------------------------------------- kernels

// K0: initial populations f = f_eq(rho, u) (u = 0 unless given), interface
// mass m = fill * sum f, fill = m / sum f
template <int S>
__global__ void k_init(Dev d, const uint8_t *flags, const double *fill, const double *rho, const double *vel) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= d.N) return;
    const int c = flags[i] & CL_MASK;
    int x, y, z;
    coords(d, i, x, y, z);
    const int fx = x == 0 || x == d.nx - 1 ? FACE_X : 0, fyz = y == 0 || y == d.ny - 1 || z == 0 || z == d.nz - 1 ? FACE_YZ : 0;
    d.flags[i] = (uint8_t)(c | fx | fyz | (d.walls_move && (fx | fyz) ? MOVING_FACE : 0));
    d.bid[i] = 0;
    d.cmark[i] = 0;
    if (c == CL_O) d.status[3] = 1;
    if (c != CL_L && c != CL_I) return;
    double u[3] = {0.0, 0.0, 0.0};
    if (vel) {
        u[0] = vel[3 * i];
        u[1] = vel[3 * i + 1];
        u[2] = vel[3 * i + 2];
    }
    double f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q] = feq_d(q, rho[i], u);
    Sto<S>::st_cell(d.fsrc, i, d.N, f);
    if (c == CL_I) {
        double r = cell_density<S>(d, d.fsrc, i);
        double m = fill[i] * r;
        d.m[i] = m;
        d.phisrc[i] = m / r;
        if constexpr (S != 0) d.phifsrc[i] = (float)(m / r);
    }
}

// the initial interface cells as the first step's list (d.list, d.cnt: those
// of the step before the first)
__global__ void k_list_interface(Dev d) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    wl_append(d, i < d.N && clsv(d, i) == CL_I, WL_IFACE, (uint32_t)i);
}

// rotation matrix and the cell range that may lie inside the body
__device__ void body_bounds(const Dev &d, Body &b) {
    rotation(b.q, b.R);
    for (int k = 0; k < 3; ++k) {
        const double fl = floor(b.o[k]);
        b.oi[k] = (int)fl;
        b.of[k] = (float)(b.o[k] - fl);  // o - floor(o) is exact in double
        b.hf[k] = (float)(b.shape == 1 && k == 0 ? b.h[0] * b.h[0] : b.h[k]);
    }
    for (int k = 0; k < 9; ++k) b.Rf[k] = (float)b.R[k];
    int n[3] = {d.nx, d.ny, d.nz};
    for (int k = 0; k < 3; ++k) {
        double e = b.shape == 1 ? b.h[0]
                                : (fabs(b.R[k * 3 + 0]) * b.h[0] + fabs(b.R[k * 3 + 1]) * b.h[1]) + fabs(b.R[k * 3 + 2]) * b.h[2];
        int lo = (int)floor(b.o[k] - e) - 1;
        int hi = (int)floor(b.o[k] + e) + 2;
        if (!(d.periodic & (1u << k))) {
            lo = lo < 0 ? 0 : lo;
            hi = hi > n[k] ? n[k] : hi;
        } else if (hi - lo > n[k]) {
            hi = lo + n[k];
        }
        if (hi < lo) hi = lo;
        b.lo[k] = lo;
        b.hi[k] = hi;
    }
}

__global__ void k_body_prepare(Dev d, int bi) {
    if (threadIdx.x != 0) return;
    Body &b = d.bodies[bi];
    body_bounds(d, b);
    // volume, mass and principal moments, every operation rounded by itself as
    // in the rigid-body update's unit
    const double *h = b.h;
    if (b.shape == 1) {  // sphere: V = 4/3 pi r^3, I = 2/5 m r^2
        b.vol = __dmul_rn(4.1887902047863905, __dmul_rn(__dmul_rn(h[0], h[0]), h[0]));
        b.mass = __dmul_rn(b.dens, b.vol);
        b.I[0] = b.I[1] = b.I[2] = __dmul_rn(__dmul_rn(0.4, b.mass), __dmul_rn(h[0], h[0]));
    } else {
        b.vol = __dmul_rn(__dmul_rn(__dmul_rn(8.0, h[0]), h[1]), h[2]);
        b.mass = __dmul_rn(b.dens, b.vol);
        const double m3 = __ddiv_rn(b.mass, 3.0);
        const double s0 = __dmul_rn(h[0], h[0]), s1 = __dmul_rn(h[1], h[1]), s2 = __dmul_rn(h[2], h[2]);
        b.I[0] = __dmul_rn(m3, __dadd_rn(s1, s2));
        b.I[1] = __dmul_rn(m3, __dadd_rn(s0, s2));
        b.I[2] = __dmul_rn(m3, __dadd_rn(s0, s1));
    }
    for (int k = 0; k < 3; ++k) {
        b.plo[k] = b.lo[k];
        b.phi[k] = b.hi[k];
    }
}

// iterate the cells of a box range [lo, hi) (wrapped on periodic axes)
__device__ __forceinline__ long long range_count(const int *lo, const int *hi) {
    return (long long)(hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2]);
}
__device__ __forceinline__ void range_cell(const Dev &d, const int *lo, const int *hi, long long k, int &x, int &y,
                                           int &z) {
    // a range holds at most the grid's cells (fewer than 2^32)
    const uint32_t lx = (uint32_t)(hi[0] - lo[0]), ly = (uint32_t)(hi[1] - lo[1]);
    const uint32_t kk = (uint32_t)k, r = kk / lx, rz = r / ly;
    x = lo[0] + (int)(kk - r * lx);
    y = lo[1] + (int)(r - rz * ly);
    z = lo[2] + (int)rz;
    if (x < 0 || x >= d.nx) x = ((x % d.nx) + d.nx) % d.nx;  // only periodic axes can leave [0, n)
    if (y < 0 || y >= d.ny) y = ((y % d.ny) + d.ny) % d.ny;
    if (z < 0 || z >= d.nz) z = ((z % d.nz) + d.nz) % d.nz;
}

// the cells of the body's range and one beyond it (all that may have an
// obstacle of the body among their neighbours)
__device__ __forceinline__ void near_range(const Dev &d, const Body &b, int *lo, int *hi) {
    const int n3[3] = {d.nx, d.ny, d.nz};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = b.lo[k] - 1;
        hi[k] = b.hi[k] + 1;
        if (!(d.periodic & (1u << k))) {
            lo[k] = lo[k] < 0 ? 0 : lo[k];
            hi[k] = hi[k] > n3[k] ? n3[k] : hi[k];
        } else if (hi[k] - lo[k] > n3[k]) {
            hi[k] = lo[k] + n3[k];
        }
        if (hi[k] < lo[k]) hi[k] = lo[k];  // a body that has left the grid through a wall has no cells
    }
}

// mapping of a newly added body (Sec. 2.3); book_mass: charge the covered mass
template <int S>
__global__ void k_map_body(Dev d, int bi, int book_mass) {
    const Body &b = d.bodies[bi];
    long long n = range_count(b.lo, b.hi);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        range_cell(d, b.lo, b.hi, k, x, y, z);
        long long i = x + (long long)d.nx * (y + (long long)d.ny * z);
        int c = clsv(d, i);
        if (c == CL_O || !inside(d, b, x, y, z)) continue;
        if (book_mass) {
            double mass = c == CL_L ? cell_density<S>(d, d.fsrc, i) : (c == CL_I ? d.m[i] : 0.0);
            if (mass != 0.0) atomicAdd(&d.ledger[LG_COVERED], mass);
        }
        set_cls(d, i, CL_O);
        d.bid[i] = (uint8_t)bi;
    }
}

// Coordinates a kernel body runs at: its launch's own block, or one entry of
// a packed block table when a single launch serves many tanks
struct VB {
    unsigned x, y, z, nx, ny, nz, kind;
};
__device__ __forceinline__ VB vb_own() {
    return VB{blockIdx.x, blockIdx.y, blockIdx.z, gridDim.x, gridDim.y, gridDim.z, 0};
}

// A worklist's items spread over a launch's blocks, a warp's worth (`per` items)
// at a time.  A short list goes to as many blocks (SMs) as possible: its
// latency chains and its double operations, each of which holds a scheduler
// for 64 cycles, don't queue behind one another.  From a group per SM up the
// blocks fill their warps, so that a long list's blocks are few and full and
// keep neighbouring items together.  First item of the calling warp and
// the stride; a warp without items starts at n.
__device__ __forceinline__ void list_span(const VB &vb, uint32_t n, uint32_t per, uint32_t &first, uint32_t &stride) {
    const uint32_t wpb = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const uint32_t groups = (n + per - 1) / per, wide = min(vb.nx, 152u), used = min(wpb, (groups + wide - 1) / wide);
    first = warp < used ? (vb.x * used + warp) * per : n;
    stride = vb.nx * used * per;
}
#define LIST_LOOP(L, var)                                                                                     \
    const uint32_t n_##var = wl_count(d, L);                                                                   \
    uint32_t f_##var, s_##var;                                                                                 \
    list_span(vb, n_##var, 32u, f_##var, s_##var);                                                             \
    for (uint32_t it_##var = f_##var + (threadIdx.x & 31u); it_##var < n_##var; it_##var += s_##var)

// Walk over the cells around a body (its range of ncell cells, lo .. hi) that
// satisfy `want(flag byte)`, by `blocks` blocks.  Few cells of the range are
// next to the body's surface, and those come in whole rows and planes: groups
// of G cells are dealt out to the blocks in turn, and a block first looks
// through the flags of its groups (CHUNK cells at a time) and packs the cells
// it wants into shared memory, then works on them with full warps
// (`work(x, y, z, i)`).
constexpr uint32_t CHUNK = 1024;
// The force kernel's blocks: on a single tank one thread per cell of a group (a
// block's group may lie wholly in a face of the body: 128^3 heeled box 34 us
// with 128 threads, 24 with 256); in a batch, where most of a group's cells are
// passed over, smaller ones so that more groups are resident.
constexpr int FORCE_THREADS = 256, FORCE_THREADS_BATCH = 128;
template <uint32_t G, class Want, class Work>
__device__ __forceinline__ void walk_near(const Dev &d, const int *lo, const int *hi, uint32_t ncell, const VB &vb,
                                          uint32_t blocks, Want want, Work work) {
    __shared__ uint32_t s_cell[CHUNK];
    __shared__ uint32_t s_n;
    if (vb.x >= blocks) return;
    const uint32_t nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31u;
    const uint32_t groups = (ncell + G - 1) / G;
    const uint32_t mine = groups > vb.x ? (groups - vb.x + blocks - 1) / blocks * G : 0;  // cells of this block
    constexpr int U = 4;  // flag loads in flight per thread
    for (uint32_t c0 = 0; c0 < mine; c0 += CHUNK) {
        const uint32_t c1 = min(c0 + CHUNK, mine);
        if (tid == 0) s_n = 0;
        __syncthreads();
        for (uint32_t l0 = c0 + tid - lane; l0 < c1; l0 += U * nthr) {  // warp-uniform
            uint32_t k[U];
            int fb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t l = l0 + u * nthr;
                k[u] = (l / G * blocks + vb.x) * G + l % G + lane;  // l: a multiple of 32
                fb[u] = 0;
                if (l < c1 && k[u] < ncell) {
                    int x, y, z;
                    range_cell(d, lo, hi, k[u], x, y, z);
                    fb[u] = d.flags[x + (long long)d.nx * (y + (long long)d.ny * z)];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool on = want(fb[u]);
                const unsigned m = __ballot_sync(0xffffffffu, on);
                uint32_t at = 0;
                if (lane == 0 && m) at = atomicAdd(&s_n, (uint32_t)__popc(m));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (on) s_cell[at + __popc(m & ((1u << lane) - 1u))] = k[u];
            }
        }
        __syncthreads();
        const uint32_t n = s_n;
        for (uint32_t j = tid; j < n; j += nthr) {
            int x, y, z;
            range_cell(d, lo, hi, s_cell[j], x, y, z);
            work(x, y, z, x + (long long)d.nx * (y + (long long)d.ny * z));
        }
        __syncthreads();
    }
}

// Blocks for a body's cells when the blocks' sums do not matter: in a batch
// (dense), whose tanks fill the GPU, as many as have CHUNK cells each, so that
// the packed warps are full; for a single tank all that fit the GPU with the
// other bodies' (two per SM), so that the work of a small body spreads.
__device__ __forceinline__ uint32_t near_blocks(const Dev &d, const VB &vb, uint32_t ncell, bool dense) {
    const uint32_t full = (ncell + CHUNK - 1) / CHUNK;
    return min(vb.nx, dense ? full : max(full, 304u / (uint32_t)d.nb));
}

// neighbour-obstacle bit: set when any of the 18 neighbours is an obstacle
// (the bulk kernel then leaves a liquid cell to k_near; walls and periodic
// seams have their own bits, set at creation)
__device__ __forceinline__ void nb_refresh(const Dev &d, long long i) {
    int x, y, z;
    coords(d, i, x, y, z);
    bool nb = false;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        int c = cls(d, nbr(d, x, y, z, cx(q), cy(q), cz(q)));
        nb = nb || c == CL_O;
    }
    d.flags[i] = (uint8_t)((d.flags[i] & ~NB_OBST) | (nb ? NB_OBST : 0));
}

// neighbour-obstacle bits of the cells x0 <= x < x1 (grid (x-tiles, ny, nz))
__global__ void k_nb_all(Dev d) {
    int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= d.nx) return;
    long long i = x + (long long)d.nx * (y + (long long)d.ny * z);
    bool nb = false;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        int c = cls(d, nbr(d, x, y, z, cx(q), cy(q), cz(q)));
        nb = nb || c == CL_O;
    }
    d.flags[i] = (uint8_t)((d.flags[i] & ~NB_OBST) | (nb ? NB_OBST : 0));
}

// the same over the cells around body bi (its range widened by one cell)
__global__ void k_nb_body(Dev d, int bi) {
    const Body &b = d.bodies[bi];
    int lo[3] = {b.lo[0] - 1, b.lo[1] - 1, b.lo[2] - 1}, hi[3] = {b.hi[0] + 1, b.hi[1] + 1, b.hi[2] + 1};
    int n3[3] = {d.nx, d.ny, d.nz};
    for (int k = 0; k < 3; ++k) {
        if (!(d.periodic & (1u << k))) {
            lo[k] = lo[k] < 0 ? 0 : lo[k];
            hi[k] = hi[k] > n3[k] ? n3[k] : hi[k];
        } else if (hi[k] - lo[k] > n3[k]) {
            hi[k] = lo[k] + n3[k];
        }
    }
    for (int zz = lo[2] + (int)blockIdx.x; zz < hi[2]; zz += gridDim.x) {
        int z = zz < 0 ? zz + d.nz : (zz >= d.nz ? zz - d.nz : zz);
        for (int yy = lo[1] + (int)threadIdx.y; yy < hi[1]; yy += blockDim.y) {
            int y = yy < 0 ? yy + d.ny : (yy >= d.ny ? yy - d.ny : yy);
            for (int xx = lo[0] + (int)threadIdx.x; xx < hi[0]; xx += blockDim.x) {
                int x = xx < 0 ? xx + d.nx : (xx >= d.nx ? xx - d.nx : xx);
                nb_refresh(d, x + (long long)d.nx * (y + (long long)d.ny * z));
            }
        }
    }
}

// the calling lane's neighbour of (x, y, z): direction = lane; -1 beyond a wall
// and for the lanes without a direction
__device__ __forceinline__ long long lane_nbr(const Dev &d, int lane, int x, int y, int z) {
    return lane >= 1 && lane < Q ? nbr(d, x, y, z, dir_x(lane), dir_y(lane), dir_z(lane)) : -1;
}
// Cells whose obstacle status changed this step (covered, uncovered): the bit
// of each and of its 18 neighbours is refreshed.
// A warp per (listed cell, direction): the target is the cell itself (q = 0) or
// its neighbour in direction q, lane p looks at the target's neighbour p; for
// long lists, of which each warp would take more than NB_WARP in turn, a thread
// per target.  Targets refreshed twice get the same value (the classes do not
// change in this kernel).  Measured, us, four 96^3 tanks of a batch with about
// 18000 targets each (on 18 blocks): 99 and 26.
#ifndef LBMFS_NB_WARP
#define LBMFS_NB_WARP 8
#endif
constexpr uint32_t NB_WARP = LBMFS_NB_WARP;
__device__ __forceinline__ long long nb_target(const Dev &d, uint32_t it, uint32_t nc) {
    const uint32_t e = it / Q;
    const int q = (int)(it - e * Q);
    const long long c = e < nc ? (long long)d.list[WL_COVER][e] : (long long)d.list[WL_PEND][e - nc];
    if (q == 0) return c;
    int x, y, z;
    coords(d, c, x, y, z);
    return nbr(d, x, y, z, dir_x(q), dir_y(q), dir_z(q));
}
__device__ __forceinline__ void nb_update_body(const Dev &d, const VB &vb) {
    if (d.nb > 1) {
        LIST_LOOP(WL_COVER, a) d.cmark[d.list[WL_COVER][it_a]] = 0;
    }
    const uint32_t nc = wl_count(d, WL_COVER), n = (nc + wl_count(d, WL_PEND)) * Q;
    const uint32_t warps = vb.nx * (blockDim.x >> 5);
    const int lane = threadIdx.x & 31;
    if (n > NB_WARP * warps) {
        for (uint32_t it = vb.x * blockDim.x + threadIdx.x; it < n; it += vb.nx * blockDim.x) {
            const long long t = nb_target(d, it, nc);
            if (t >= 0) nb_refresh(d, t);
        }
        return;
    }
    for (uint32_t it = (threadIdx.x >> 5) * vb.nx + vb.x; it < n; it += warps) {
        const long long t = nb_target(d, it, nc);
        if (t < 0) continue;
        int x, y, z;
        coords(d, t, x, y, z);
        const bool obst = cls(d, lane_nbr(d, lane, x, y, z)) == CL_O;
        const bool nb = __any_sync(0xffffffffu, obst);
        if (lane == 0) d.flags[t] = (uint8_t)((d.flags[t] & ~NB_OBST) | (nb ? NB_OBST : 0));
        __syncwarp();
    }
}

// ---- C4: momentum exchange at the links into body vb.y (state at t):
// Sec. 2.3 Eqs. momentumexchange, netforce, torque; Sec. 2.4 Eq.
// momentuminterface for interface cells
// Fixed-point sums of the float storages' per-cell force remainders: v * 2^s
// rounded to nearest (ties away from zero), built from the float's bits with
// integer operations (no double arithmetic; integer sums are exact, so the
// block and body totals do not depend on the order of the cells).
// |v| >= 2^(62 - s) (and a non-finite v) saturates at 2^62 in magnitude.
constexpr int FX_FORCE = 32, FX_TORQUE = 30;
__device__ __forceinline__ long long fixed_point(float v, int s) {
    const unsigned b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xffu);
    const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
    const int sh = e - 150 + s;  // |v| 2^s = m 2^sh for normal numbers
    long long r;
    if (e == 0 || sh < -25) r = 0;
    else if (sh < 0) r = (m + (1ll << (-sh - 1))) >> -sh;
    else r = sh > 38 ? (1ll << 62) : (m << sh);
    return (b >> 31) ? -r : r;
}

// Double-precision sums of Eqs. netforce and torque, exact and independent of
// the order of the terms: a term t (|t| < 2^31) becomes the integer
// floor(t 2^96) (its bits below 2^-96 dropped) and the integers are added in
// 128-bit two's complement; the total v = H 2^64 + L (H signed, L unsigned)
// becomes the double H 2^-32 + L 2^-96.  The plain CPU restatement sums the
// same way, so both give the same bits whatever the thread order.
__device__ __forceinline__ unsigned __int128 fixed96(double t) {
    const double sc = t * 4294967296.0;  // t 2^32, exact
    const double hf = floor(sc);
    const long long hi = (long long)hf;
    const unsigned long long lo = (unsigned long long)((sc - hf) * 18446744073709551616.0);
    return ((unsigned __int128)(unsigned long long)hi << 64) | (unsigned __int128)lo;
}
__device__ __forceinline__ double fixed96_value(unsigned __int128 v) {
    const long long H = (long long)(unsigned long long)(v >> 64);
    const unsigned long long L = (unsigned long long)v;
    return (double)H * 2.3283064365386962890625e-10 + (double)L * 1.2621774483536188886587657044524580e-29;
}
__device__ __forceinline__ unsigned __int128 shfl_xor_128(unsigned __int128 v, int off) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, off);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), off);
    return ((unsigned __int128)hi << 64) | (unsigned __int128)lo;
}
__device__ __forceinline__ unsigned __int128 shfl_down_128(unsigned __int128 v, int off) {
    const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)v, off);
    const unsigned long long hi = __shfl_down_sync(0xffffffffu, (unsigned long long)(v >> 64), off);
    return ((unsigned __int128)hi << 64) | (unsigned __int128)lo;
}

template <int S, bool DENSE>
__device__ __forceinline__ void forces_f64_body(const Dev &d, const VB &vb) {
    const int bi = vb.y;
    const Body &b = d.bodies[bi];
    unsigned __int128 acc[7] = {0, 0, 0, 0, 0, 0, 0};
    // only cells next to an obstacle (neighbour-obstacle bit) can hold links
    const long long sy = d.nx, sz = (long long)d.nx * d.ny;
    int lo[3], hi[3];
    near_range(d, b, lo, hi);
    const uint32_t ncell = (uint32_t)range_count(lo, hi);
    walk_near<32>(d, lo, hi, ncell, vb, near_blocks(d, vb, ncell, DENSE), [](int fb) { return (fb & NB_OBST) && (fb & CL_MASK) != CL_O; },
                  [&](int x, int y, int z, long long i) {
        const int cl = clsv(d, i);
        // directions into body bi and the cell's populations, requested at once
        const bool inner = x > 0 && x < d.nx - 1 && y > 0 && y < d.ny - 1 && z > 0 && z < d.nz - 1;
        const bool fluid = cl != CL_G;
        double f[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) f[q] = fluid ? Sto<S>::ldf(d.fsrc, q, i, d.N) : 0.0;
        const double phi_x = cl == CL_L ? 1.0 : (cl == CL_I ? d.phisrc[i] : 0.0);
        unsigned lm = 0;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const long long si = inner ? i - (cx(q) + cy(q) * sy + cz(q) * sz) : nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
            if (si >= 0 && clsv(d, si) == CL_O) lm |= 1u << q;
        }
        if (d.nb > 1) {
            unsigned om = lm;
            lm = 0;
#pragma unroll
            for (int q = 1; q < Q; ++q)
                if (om & (1u << q)) {
                    const long long si =
                        inner ? i - (cx(q) + cy(q) * sy + cz(q) * sz) : nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
                    if (d.bid[si] == bi) lm |= 1u << q;
                }
        }
        if (!lm) return;
        // double, each value in the order of the plain restatement; the
        // direction is a constant of each unrolled term, so products by its
        // zeros are left out (x + 0 y = x)
        const double r[3] = {min_image(d, (x + 0.5) - b.o[0], 0), min_image(d, (y + 0.5) - b.o[1], 1),
                             min_image(d, (z + 0.5) - b.o[2], 2)};
        double rho_x = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) rho_x += f[q];
        const double pg = 1.0 - phi_x;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            if (!(lm & (1u << q))) continue;
            const int qb = opp(q);
            double inr = wd(q) * d.rho_g;
            if (fluid) {
                const double cuw = link_cuw(d, b, x, y, z, q);
                const double A = phi_x * f[qb], B = pg * inr;
                const double C = cuw == 0.0 ? 0.0 : phi_x * (((3.0 * wd(q)) * rho_x) * cuw);
                inr = (A + B) + C;
            }
            const double g = 2.0 * inr;
            // the integer of +-g: floor(-t) = -floor(t) where t 2^96 is an
            // integer, which holds from |g| = 2^-43 up
            const unsigned __int128 pos = fixed96(g);
            const unsigned __int128 neg = fabs(g) >= 1.1368683772161603e-13 ? (unsigned __int128)0 - pos : fixed96(-g);
            if (cx(qb)) acc[0] += cx(qb) > 0 ? pos : neg;
            if (cy(qb)) acc[1] += cy(qb) > 0 ? pos : neg;
            if (cz(qb)) acc[2] += cz(qb) > 0 ? pos : neg;
            const double F0 = cx(qb) > 0 ? g : -g, F1 = cy(qb) > 0 ? g : -g, F2 = cz(qb) > 0 ? g : -g;
            if (cy(qb) && cz(qb)) acc[3] += fixed96(r[1] * F2 - r[2] * F1);
            else if (cz(qb)) acc[3] += fixed96(r[1] * F2);
            else if (cy(qb)) acc[3] += fixed96(-(r[2] * F1));
            if (cx(qb) && cz(qb)) acc[4] += fixed96(r[2] * F0 - r[0] * F2);
            else if (cx(qb)) acc[4] += fixed96(r[2] * F0);
            else if (cz(qb)) acc[4] += fixed96(-(r[0] * F2));
            if (cx(qb) && cy(qb)) acc[5] += fixed96(r[0] * F1 - r[1] * F0);
            else if (cy(qb)) acc[5] += fixed96(r[0] * F1);
            else if (cx(qb)) acc[5] += fixed96(-(r[1] * F0));
            acc[6] += g >= 0.0 ? pos : neg;
        }
    });
    // block reduction of the exact integer sums (any order gives the same
    // bits); a warp without any link skips the tree (its sums are zeros).
    // The block's partials go out as 128-bit integers (low, high word).
    __shared__ unsigned __int128 sh[FORCE_THREADS / 32][7];
    const int tid = threadIdx.x;
    int lane = tid & 31, wid = tid >> 5;
    const bool any = __any_sync(0xffffffffu, (acc[6] | acc[0] | acc[1] | acc[2]) != 0);
#pragma unroll
    for (int c = 0; c < 7; ++c) {
        unsigned __int128 v = acc[c];
        if (any)
            for (int off = 16; off > 0; off >>= 1) v += shfl_down_128(v, off);
        if (lane == 0) sh[wid][c] = v;
    }
    __syncthreads();
    if (tid < 7) {
        unsigned __int128 v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sh[w][tid];
        unsigned long long *p = reinterpret_cast<unsigned long long *>(d.part) +
                                2 * (((long long)bi * FORCE_BLOCKS + vb.x) * 7 + tid);
        p[0] = (unsigned long long)v;
        p[1] = (unsigned long long)(v >> 64);
    }
}

// Sum of a 64-bit integer over the 32 lanes of a warp: three limbs (bits
// 0-20, 21-41 and the signed rest) summed by warp reductions, whose 32-lane
// sums stay within 32 bits for |v| < 2^62.
__device__ __forceinline__ long long warp_sum64(long long v) {
    const unsigned c = (unsigned)(v & 0x1fffffll), b = (unsigned)((v >> 21) & 0x1fffffll);
    const int a = (int)(v >> 42);
    const unsigned sc = __reduce_add_sync(0xffffffffu, c), sb = __reduce_add_sync(0xffffffffu, b);
    const int sa = __reduce_add_sync(0xffffffffu, a);
    return (long long)sa * (1ll << 42) + (long long)sb * (1ll << 21) + (long long)sc;
}

// Float storages.  Every sum within a block is an integer, so a block's totals
// do not depend on the cell-to-thread map; which cells a block sums is fixed
// (FORCE_GROUP consecutive cells of the range, dealt out to as many blocks as
// there are groups), so the totals are the same in every launch form.  The
// link term is split into the uniform gas-pressure part 2 w_q rho_G (exact
// integer sums of 36 (2 w_q) c_qbar and of the lever arm twice the cell centre)
// and the small remainder 2 (phi (f_qbar - w_q rho_G) + moving-wall part),
// computed in float from the stored deviations f - w and summed in fixed point.
// The lever arm r is the cell's, so each part is summed over the cell's links
// first and its torque is r x that sum.
constexpr uint32_t FORCE_GROUP = 256;
template <int S, bool DENSE>
__device__ __forceinline__ void forces_float_body(const Dev &d, const VB &vb) {
    const int bi = vb.y;
    const Body &b = d.bodies[bi];
    const int n3[3] = {d.nx, d.ny, d.nz};
    long long ia[7] = {0, 0, 0, 0, 0, 0, 0};         // fixed-point remainder sums
    long long ik[3] = {0, 0, 0}, it[3] = {0, 0, 0};  // exact gas-pressure sums
    bool hit = false;
    // body state in float, rounded once per thread
    const float of[3] = {(float)b.o[0], (float)b.o[1], (float)b.o[2]};
    const float vf[3] = {(float)b.v[0], (float)b.v[1], (float)b.v[2]};
    const float wfv[3] = {(float)b.w[0], (float)b.w[1], (float)b.w[2]};
    const float rg = (float)d.rho_g, wrg1 = d.rg1_f;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarp = blockDim.x >> 5;
    const long long sy = d.nx, sz = (long long)d.nx * d.ny;
    int lo[3], hi[3];
    near_range(d, b, lo, hi);
    const uint32_t ncell = (uint32_t)range_count(lo, hi);
    const uint32_t used = min(vb.nx, (ncell + FORCE_GROUP - 1) / FORCE_GROUP);
    if (vb.x >= used) {  // the others contribute zeros
        if (tid < 7) d.part[((long long)bi * FORCE_BLOCKS + vb.x) * 7 + tid] = 0.0;
        return;
    }
    walk_near<FORCE_GROUP>(d, lo, hi, ncell, vb, used, [](int fb) { return (fb & NB_OBST) && (fb & CL_MASK) != CL_O; },
                           [&](int x, int y, int z, long long i) {
            const int cl = clsv(d, i);
            // directions into body bi: all neighbour classes requested at
            // once (linear offsets away from the grid faces), then the body
            // ids of the obstacle directions
            const bool inner = x > 0 && x < d.nx - 1 && y > 0 && y < d.ny - 1 && z > 0 && z < d.nz - 1;
            // a liquid or interface cell's link terms read its populations:
            // requested together with the neighbour classes
            float fc[Q];
            if (cl != CL_G) {
#pragma unroll
                for (int q = 0; q < Q; ++q) fc[q] = Sto<S>::ld(d.fsrc, q, i, d.N);
            }
            unsigned om = 0;
#pragma unroll
            for (int q = 1; q < Q; ++q) {
                const long long si = inner ? i - (cx(q) + cy(q) * sy + cz(q) * sz)
                                           : nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
                if (si >= 0 && clsv(d, si) == CL_O) om |= 1u << q;
            }
            unsigned lm = om;  // with one body every obstacle cell is its
            if (d.nb > 1) {
                lm = 0;
#pragma unroll
                for (int q = 1; q < Q; ++q)
                    if (om & (1u << q)) {
                        const long long si = inner ? i - (cx(q) + cy(q) * sy + cz(q) * sz)
                                                   : nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
                        if (d.bid[si] == bi) lm |= 1u << q;
                    }
            }
            if (!lm) return;
            hit = true;
            const float phf = cl == CL_L ? 1.0f : (cl == CL_I ? d.phifsrc[i] : 0.0f);
            // lever arm from the cell centre (minimum image on periodic
            // axes): float for the small remainder, and twice the cell
            // centre as an integer for the exact gas-pressure part
            const int xyz[3] = {x, y, z};
            float rf[3];
            long long c2[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                int xk = xyz[k];
                rf[k] = ((float)xk + 0.5f) - of[k];
                if (d.periodic & (1u << k)) {
                    const int shn = (int)floorf(rf[k] / (float)n3[k] + 0.5f);
                    xk -= shn * n3[k];
                    rf[k] -= (float)(shn * n3[k]);
                }
                c2[k] = 2ll * xk + 1;
            }
            float rho_x = -1.0f;
            int kx = 0, ky = 0, kz = 0;  // sum of 36 (2 w_q) c_qbar over the links
            float gx = 0.0f, gy = 0.0f, gz = 0.0f, fabs_sum = 0.0f;
#pragma unroll
            for (int q = 1; q < Q; ++q) {
                if (!(lm & (1u << q))) continue;
                const int qb = opp(q);
                const int m36 = q <= 6 ? 4 : 2;  // 36 x 2 w_q
                float gdev = 0.0f;
                if (cl != CL_G) {
                    // u_w at the link midpoint, r + c_qbar / 2 from the body centre
                    const float px = rf[0] + 0.5f * cx(qb), py = rf[1] + 0.5f * cy(qb), pz = rf[2] + 0.5f * cz(qb);
                    const float ux = vf[0] + (wfv[1] * pz - wfv[2] * py);
                    const float uy = vf[1] + (wfv[2] * px - wfv[0] * pz);
                    const float uz = vf[2] + (wfv[0] * py - wfv[1] * px);
                    const float cuw = cx(q) * ux + cy(q) * uy + cz(q) * uz;
                    float C = 0.0f;
                    if (cuw != 0.0f) {
                        if (rho_x < 0.0f) {
                            float dr = 0.0f;
#pragma unroll
                            for (int k = 0; k < Q; ++k) dr += fc[k];
                            rho_x = 1.0f + dr;
                        }
                        C = phf * (3.0f * wf(q) * rho_x * cuw);
                    }
                    const float dev = fc[qb] + wf(q) * wrg1;
                    gdev = 2.0f * (phf * dev + C);
                }
                if (cx(qb)) {
                    kx += cx(qb) * m36;
                    gx += cx(qb) * gdev;
                }
                if (cy(qb)) {
                    ky += cy(qb) * m36;
                    gy += cy(qb) * gdev;
                }
                if (cz(qb)) {
                    kz += cz(qb) * m36;
                    gz += cz(qb) * gdev;
                }
                fabs_sum += fabsf((float)m36 * (rg * (1.0f / 36.0f)) + gdev);
            }
            ia[0] += fixed_point(gx, FX_FORCE);
            ia[1] += fixed_point(gy, FX_FORCE);
            ia[2] += fixed_point(gz, FX_FORCE);
            ia[3] += fixed_point(rf[1] * gz - rf[2] * gy, FX_TORQUE);
            ia[4] += fixed_point(rf[2] * gx - rf[0] * gz, FX_TORQUE);
            ia[5] += fixed_point(rf[0] * gy - rf[1] * gx, FX_TORQUE);
            ia[6] += fixed_point(fabs_sum, FX_FORCE);
            // gas-pressure part (rho_G / 36) K: its torque is
            // (rho_G / 36) (sum c2 x K / 2 - o x sum K)
            ik[0] += kx;
            ik[1] += ky;
            ik[2] += kz;
            it[0] += c2[1] * kz - c2[2] * ky;
            it[1] += c2[2] * kx - c2[0] * kz;
            it[2] += c2[0] * ky - c2[1] * kx;
    });
    // warp sums, then the warps' sums in the block (integers: exact); a warp
    // without any link skips the reductions (its sums are zeros)
    __shared__ long long shi[FORCE_THREADS / 32][13];
    const bool any = __any_sync(0xffffffffu, hit);
#pragma unroll
    for (int c = 0; c < 13; ++c) {
        long long v = c < 7 ? ia[c] : (c < 10 ? ik[c - 7] : it[c - 10]);
        if (any) v = warp_sum64(v);
        if (lane == 0) shi[wid][c] = any ? v : 0ll;
    }
    __syncthreads();
    if (tid < 7) {
        long long I = 0;
        for (int w = 0; w < nwarp; ++w) I += shi[w][tid];
        double v = (double)I * (tid >= 3 && tid < 6 ? 1.0 / (double)(1ll << FX_TORQUE) : 1.0 / (double)(1ll << FX_FORCE));
        if (tid < 6) {
            long long K[3] = {0, 0, 0}, T2[3] = {0, 0, 0};
            for (int w = 0; w < nwarp; ++w)
                for (int k = 0; k < 3; ++k) {
                    K[k] += shi[w][7 + k];
                    T2[k] += shi[w][10 + k];
                }
            const double g36 = d.rho_g / 36.0;
            if (tid < 3) {
                v += g36 * (double)K[tid];
            } else {
                const int k = tid - 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
                // (sum c2 x K) / 2 - o x sum K, component k
                const double ox = b.o[k1] * (double)K[k2] - b.o[k2] * (double)K[k1];
                v += g36 * (0.5 * (double)T2[k] - ox);
            }
        }
        d.part[((long long)bi * FORCE_BLOCKS + vb.x) * 7 + tid] = v;
    }
}

template <int S, bool DENSE>
__device__ __forceinline__ void forces_body(const Dev &d, const VB &vb) {
    if constexpr (S == 0) forces_f64_body<S, DENSE>(d, vb);
    else forces_float_body<S, DENSE>(d, vb);
}

template <int S>
__global__ void __launch_bounds__(FORCE_THREADS, S == 0 ? 2 : LBMFS_FORCE_MINB / 2) k_forces(const __grid_constant__ Dev d) {
    launch_dependents();
    forces_body<S, false>(d, vb_own());
}

// ---- C1 + C2 for liquid cells (Sec. 2.1 Eqs. stream, lbgk, forceterm;
// Sec. 2.3 Eq. noslip); interface cells are listed for the next step's k_interface
template <int S, int ZBMAX>
__device__ __forceinline__ void liquid_column(const Dev &d, bool in, int x, int y, int z0, int z1);

// A block covers BULK_THREADS consecutive cells of an xy-plane (row ends
// wrap to the next row, so narrow grids keep every lane busy) for zb
// consecutive z: grid (ceil(nx ny / BULK_THREADS), 1, ceil(nz / zb)).
template <int S, int ZBMAX>
__device__ __forceinline__ void liquid_body(const Dev &d, const VB &vb, int zb) {
    // a tile above the previous step's fluid (plus a margin) holds only gas
    if ((int)(vb.z * zb) > __ldg(d.ztop_rd) + ZTOP_MARGIN) return;
    const unsigned p = vb.x * BULK_THREADS + threadIdx.x;
    const bool in = p < (unsigned)d.nx * (unsigned)d.ny;
    const int y = in ? (int)(p / (unsigned)d.nx) : 0;
    const int x = in ? (int)p - y * d.nx : 0;
    const int z0 = vb.z * zb;
    const int z1 = min(z0 + zb, d.nz);
    liquid_column<S, ZBMAX>(d, in, x, y, z0, z1);
}
template <int S, int ZB>
__global__ void __launch_bounds__(BULK_THREADS, S == 0 ? 1 : LBMFS_BULK_MINB)
    k_liquid(const __grid_constant__ Dev d) {
    liquid_body<S, ZB>(d, vb_own(), ZB);
}

template <int S>
__device__ __forceinline__ void collide_store(const Dev &d, typename Sto<S>::R *fp, long long i) {
    using P = Sto<S>;
    if constexpr (!P::shifted) {
        double fn[Q];
        const double rho = collide_d(d, fp, fn);
        // The stored sum r has to be a positive number.  It is rho up to the
        // roundings of the collision and of the sum, below 1e-7 in all while
        // every |f| < 2^20, so it needs no adding up (18 of 329 double
        // operations) unless some population is larger or not finite -- seen in
        // the exponents, by integer operations -- or rho is small.
        int big = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            P::st(d.fdst, q, i, d.N, fn[q]);
            big = max(big, __double2hiint(fn[q]) & 0x7fffffff);
        }
        if (big >= 0x41300000 || !(rho >= 1e-6)) {  // 2^20
            double r = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) r += fn[q];
            if (!(r == r) || r <= 0.0) atomicOr(d.status, ST_NONFINITE);
        }
    } else {
        // fp in the storage's raw units (to_raw)
        void *g = d.fdst;
        const long long N = d.N;
        float rho = collide_store_v<P::SCALE, false, float>(d, fp, [&](int q, float v) { return P::st_raw(g, q, i, N, v); });
        if (!vpos_finite(rho)) atomicOr(d.status, ST_NONFINITE);
    }
}

// populations gathered as values into the storage's raw units (q >= 1 times
// the FP16 storage's scale; exact)
template <int S> __device__ __forceinline__ void to_raw(typename Sto<S>::R *fp) {
    if constexpr (S == 2) {
#pragma unroll
        for (int q = 1; q < Q; ++q) fp[q] *= F16_SCALE;
    }
}

// populations arriving at a liquid cell with an obstacle or wall neighbour, or
// on a periodic seam: per-direction source classes, bounce-back where the
// source is solid (Eq. noslip), 6 w_q rho_x c_q.u_w added where the solid
// moves.  Three rounds of independent loads: the 18 source classes with the
// cell's own 19 populations; the pulled populations with the body ids of the
// obstacle sources; the state of the body (one body for all links when they
// share it, the common case; per link otherwise).  rho_x, in double for the
// FP64 storage and in float for the float storages, sums the own populations
// in q order.  Returns the mass the moving links add to the cell (for the
// ledger).  With owner >= 0 the cell is the caller's (mine) when its obstacle
// neighbours' lowest body is `owner`.
template <int S>
__device__ __forceinline__ double gather_general(const Dev &d, int x, int y, int z, long long i,
                                                 typename Sto<S>::R *fp, int owner, bool &mine) {
    using P = Sto<S>;
    using R = typename P::R;
    const long long N = d.N;
    long long src[Q];
    int ns[Q];
    R own[Q];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        src[q] = nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
        ns[q] = src[q] < 0 ? CL_WALL : clsv(d, src[q]);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) own[q] = P::ld(d.fsrc, q, i, N);
    unsigned moving = 0, obst = 0;  // directions with a moving solid source / an obstacle source
    int bq[Q];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const bool pull = ns[q] == CL_L || ns[q] == CL_I;
        fp[q] = pull ? P::ld(d.fsrc, q, src[q], N) : own[opp(q)];
        bq[q] = ns[q] == CL_O ? d.bid[src[q]] : -1;
        if (ns[q] == CL_O) obst |= 1u << q;
        if (ns[q] == CL_O || (ns[q] == CL_WALL && d.walls_move)) moving |= 1u << q;
        if (ns[q] == CL_G) atomicOr(d.status, ST_LIQUID_GAS);
    }
    fp[0] = own[0];
    mine = true;
    if (!moving) return 0.0;
    int b0 = -1, low = MAX_BODIES;
    bool one = true;  // every obstacle link belongs to body b0
#pragma unroll
    for (int q = 1; q < Q; ++q)
        if (obst & (1u << q)) {
            if (b0 < 0) b0 = bq[q];
            one = one && bq[q] == b0;
            low = min(low, bq[q]);
        }
    if (owner >= 0 && low != owner) {
        mine = false;
        return 0.0;
    }
    R wall = 0;
    if constexpr (S == 0) {
        double rho_x = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) rho_x += own[q];
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            if (!(moving & (1u << q))) continue;
            const double cuw = (obst & (1u << q)) ? link_cuw(d, d.bodies[one ? b0 : bq[q]], x, y, z, q)
                                                  : wall_cuw(d, x, y, z, q);
            if (cuw == 0.0) continue;
            const double srcm = ((6.0 * wd(q)) * rho_x) * cuw;
            fp[q] = fp[q] + srcm;
            wall += srcm;
        }
    } else {
        float dr = 0.0f;
#pragma unroll
        for (int k = 0; k < Q; ++k) dr += own[k];
        const float rho_x = 1.0f + dr;
        BodyF bf0;
        if (b0 >= 0) bf0 = body_f(d.bodies[b0], x, y, z);
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            if (!(moving & (1u << q))) continue;
            const float cuw = (obst & (1u << q))
                                  ? (one ? link_cuw_f(d, bf0, q) : link_cuw_f(d, d.bodies[bq[q]], x, y, z, q))
                                  : (float)wall_cuw(d, x, y, z, q);
            if (cuw == 0.0f) continue;
            const float srcm = ((6.0f * wf(q)) * rho_x) * cuw;
            fp[q] = fp[q] + srcm;
            wall += srcm;
        }
    }
    return (double)wall;
}

// C1 + C2 for the liquid cells that the bulk kernel leaves out, by the general
// gather.  They read the source grid and write their own cell of the
// destination grid only, as the bulk kernel would have.  The mass the moving
// links add is summed per warp and goes to the ledger with one atomic per warp
// (thousands of cells adding to one address would queue on it).  Blocks of
// GEN_THREADS spread the few cells over many SMs.
constexpr int GEN_THREADS = 128;
__device__ __forceinline__ void book_wall(const Dev &d, double wacc) {
    if (__any_sync(0xffffffffu, wacc != 0.0)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) wacc += __shfl_xor_sync(0xffffffffu, wacc, off);
        if ((threadIdx.x & 31) == 0 && wacc != 0.0) atomicAdd(&d.ledger[LG_WALL], wacc);
    }
}
// Cells next to a body: every liquid cell with an obstacle among its
// neighbours lies in the range around that obstacle's body, so the blocks of
// body vb.y look through its range (a cell next to two bodies is the lower
// one's).  Obstacles of the initial classes may lie anywhere: in a tank with
// such (Dev::loose) the blocks look through the whole grid.  Nothing here
// depends on the bulk kernel, beside which it runs.
template <int S, bool DENSE> __device__ __forceinline__ void near_body(const Dev &d, const VB &vb) {
    const int bi = vb.y, owner = d.nb > 1 && !d.loose ? bi : -1;
    double wacc = 0.0;
    uint32_t count = 0;
    int lo[3] = {0, 0, 0}, hi[3] = {d.nx, d.ny, d.nz};
    if (!d.loose) near_range(d, d.bodies[bi], lo, hi);
    const uint32_t ncell = (uint32_t)range_count(lo, hi), blocks = d.loose ? vb.nx : near_blocks(d, vb, ncell, DENSE);
    walk_near<32>(d, lo, hi, ncell, vb, blocks, [](int fb) { return (fb & (CL_MASK | NB_OBST)) == (CL_L | NB_OBST); },
                     [&](int x, int y, int z, long long i) {
                         typename Sto<S>::R fp[Q];
                         bool mine;
                         const double wall = gather_general<S>(d, x, y, z, i, fp, owner, mine);
                         if (!mine) return;
                         to_raw<S>(fp);
                         collide_store<S>(d, fp, i);
                         wacc += wall;
                         ++count;
                     });
    book_wall(d, wacc);
    count = __reduce_add_sync(0xffffffffu, count);
    if ((threadIdx.x & 31) == 0 && count) atomicAdd(&d.cnt[CN_NEAR], count);
}
// Liquid cells on a face of a grid with moving walls and next to no obstacle:
// the bulk kernel leaves them out by their face bit, this walks the faces, each
// cell once: the first and last xy-plane, then the first and last row and
// column of the planes between.
template <int S> __device__ __forceinline__ void faces_body(const Dev &d, const VB &vb) {
    const uint32_t nx = d.nx, ny = d.ny, nz = d.nz, two_x = min(nx, 2u), two_y = min(ny, 2u), two_z = min(nz, 2u);
    const uint32_t mz = nz - two_z, my = ny - two_y;  // planes, rows between
    const uint32_t n1 = two_z * nx * ny, n2 = n1 + mz * two_y * nx, n = n2 + mz * my * two_x;
    const int lane = threadIdx.x & 31;
    uint32_t first, stride, count = 0;
    list_span(vb, n, 32u, first, stride);
    double wacc = 0.0;
    for (uint32_t k0 = first; k0 < n; k0 += stride) {
        uint32_t k = k0 + lane;
        if (k < n) {
            uint32_t x, y, z;
            if (k < n1) {
                x = k % nx;
                y = k / nx % ny;
                z = k / (nx * ny) ? nz - 1 : 0;
            } else if (k < n2) {
                k -= n1;
                x = k % nx;
                y = k / nx % two_y ? ny - 1 : 0;
                z = 1 + k / (nx * two_y);
            } else {
                k -= n2;
                x = k % two_x ? nx - 1 : 0;
                y = 1 + k / two_x % my;
                z = 1 + k / (two_x * my);
            }
            const long long i = x + (long long)nx * (y + (long long)ny * z);
            if ((d.flags[i] & (CL_MASK | NB_OBST)) == CL_L) {
                typename Sto<S>::R fp[Q];
                bool mine;
                wacc += gather_general<S>(d, (int)x, (int)y, (int)z, i, fp, -1, mine);
                to_raw<S>(fp);
                collide_store<S>(d, fp, i);
                ++count;
            }
        }
        __syncwarp();
    }
    book_wall(d, wacc);
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0 && count) atomicAdd(&d.cnt[CN_NEAR], count);
}
template <int S>
__global__ void __launch_bounds__(GEN_THREADS, 1) k_near(const __grid_constant__ Dev d) {
    near_body<S, false>(d, vb_own());
}
template <int S>
__global__ void __launch_bounds__(GEN_THREADS, 1) k_faces(const __grid_constant__ Dev d) {
    faces_body<S>(d, vb_own());
}

// The liquid cells that the bulk kernel steps: not those with the
// neighbour-obstacle bit (k_near) or on a face of a grid with moving walls
// (k_faces).  With the byte CL_L the cell is also on no
// face.
__device__ __forceinline__ bool bulk_cell(int c) { return (c & (CL_MASK | NB_OBST | MOVING_FACE)) == CL_L; }
// One such cell (class byte c, coordinates x, y, z, index i; not
// next to an obstacle): gather its 18 arriving populations by the cheapest rule
// that holds for it, collide and store.
template <int S>
__device__ __forceinline__ void liquid_one(const Dev &d, int c, int x, int y, int z, long long i) {
    using P = Sto<S>;
    using R = typename P::R;
    const long long N = d.N;
    R fp[Q];
    if (c == CL_L) {
        // no obstacle or wall in the neighbourhood and a liquid cell never
        // touches gas: plain pull from the 18 neighbours
        const long long sy = d.nx, sz = (long long)d.nx * d.ny;
#pragma unroll
        for (int q = 1; q < Q; ++q) fp[q] = P::ldg_raw(d.fsrc, q, i - (cx(q) + cy(q) * sy + cz(q) * sz), N);
        fp[0] = P::ldg_raw(d.fsrc, 0, i, N);
    } else if (!d.periodic) {
        // on a face of a grid without periodic axes, no obstacle
        // neighbour: a source beyond a face is a resting wall, which
        // returns the cell's own opposite population (Eq. noslip, u_w = 0)
        const long long sy = d.nx, sz = (long long)d.nx * d.ny;
        const bool xl = x == 0, xh = x == d.nx - 1, yl = y == 0, yh = y == d.ny - 1, zl = z == 0, zh = z == d.nz - 1;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const bool out = (cx(q) > 0 && xl) || (cx(q) < 0 && xh) || (cy(q) > 0 && yl) || (cy(q) < 0 && yh) ||
                             (cz(q) > 0 && zl) || (cz(q) < 0 && zh);
            fp[q] = out ? P::ldg_raw(d.fsrc, opp(q), i, N)
                        : P::ldg_raw(d.fsrc, q, i - (cx(q) + cy(q) * sy + cz(q) * sz), N);
        }
        fp[0] = P::ldg_raw(d.fsrc, 0, i, N);
    } else {
        // on a face with periodic axes: pull across the seams, walls as above
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const long long si = nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
            fp[q] = si >= 0 ? P::ldg_raw(d.fsrc, q, si, N) : P::ldg_raw(d.fsrc, opp(q), i, N);
        }
        fp[0] = P::ldg_raw(d.fsrc, 0, i, N);
    }
    collide_store<S>(d, fp, i);  // one copy of the collision in the kernel
}
// The cells (x, y, z0 .. z1-1) of one thread.  The flags of the whole column
// come in one round of loads, so a thread whose column holds no fluid leaves
// after one memory latency, and a fluid cell waits on its populations only.
template <int S, int ZBMAX>
__device__ __forceinline__ void liquid_column(const Dev &d, bool in, int x, int y, int z0, int z1) {
    static_assert(ZBMAX <= 8, "flags of a column (z1 - z0 <= ZBMAX) are packed into 64 bits");
    const long long sz = (long long)d.nx * d.ny;
    // (cell indices are below 2^32)
    long long i = (long long)((unsigned)x + (unsigned)d.nx * ((unsigned)y + (unsigned)d.ny * (unsigned)z0));
    uint64_t fl = 0;
#pragma unroll
    for (int k = 0; k < ZBMAX; ++k)
        if (in && z0 + k < z1) fl |= (uint64_t)d.flags[i + k * sz] << (8 * k);
    // record the highest tile holding liquid or interface cells (one atomic per warp)
    if (__any_sync(0xffffffffu, (fl & 0x0303030303030303ull) != 0) && (threadIdx.x & 31) == 0)
        atomicMax(d.ztop_wr, z1 - 1);
    if (fl == 0) return;
#pragma unroll 1
    for (int z = z0; fl != 0; ++z, i += sz) {  // up to the column's last cell with a class
        const int c = (int)(fl & 0xff);
        fl >>= 8;
        wl_append(d, (c & CL_MASK) == CL_I, WL_IFACE, (uint32_t)i);
        if (!bulk_cell(c)) continue;
        liquid_one<S>(d, c, x, y, z, i);  // one copy of the collision in the kernel
    }
}

// ---------------------------------------- software-pipelined bulk kernel
//
// Each thread copies the 19 populations its cell will pull at the next z into
// private shared-memory slots with cp.async (4-byte copies, no register held
// while in flight) before it collides the cell at the current z: two planes of
// loads in flight per thread.  A thread reads only its own slots, so no block
// barrier is needed; cp.async.wait_group orders the copies with the reads.
// FP16 storage copies the aligned 4-byte word holding the wanted half.

__device__ __forceinline__ void cp_async4(void *smem_dst, const void *gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int S> struct Pipe;
template <> struct Pipe<1> {
    static __device__ __forceinline__ const void *src(const Dev &d, int q, long long e) {
        return reinterpret_cast<const float *>(d.fsrc) + (long long)q * d.N + e;
    }
    static __device__ __forceinline__ float get(const uint32_t *slot, int q, long long, long long) {
        return __uint_as_float(slot[q * BULK_THREADS]);
    }
};
template <> struct Pipe<2> {
    static __device__ __forceinline__ const void *src(const Dev &d, int q, long long e) {
        if (q == 0) return reinterpret_cast<const float *>(d.fsrc) + e;
        const __half *h = reinterpret_cast<const __half *>(reinterpret_cast<const float *>(d.fsrc) + d.N) +
                          (long long)(q - 1) * d.N + e;
        return reinterpret_cast<const void *>(reinterpret_cast<uintptr_t>(h) & ~(uintptr_t)3);
    }
    static __device__ __forceinline__ float get(const uint32_t *slot, int q, long long e, long long N) {
        uint32_t w = slot[q * BULK_THREADS];
        if (q == 0) return __uint_as_float(w);
        // the half planes start 4-byte aligned; the parity of the half's index
        // counted from there picks the half within the copied word
        long long h = (long long)(q - 1) * N + e;
        unsigned short hb = (unsigned short)((h & 1) ? (w >> 16) : (w & 0xffffu));
        return __half2float(__ushort_as_half(hb)) * F16_INV_SCALE;
    }
};

template <int S>
__global__ void __launch_bounds__(BULK_THREADS, LBMFS_BULK_MINB) k_liquid_pipe(Dev d) {
    // this variant visits every tile: record the grid's top so the next step skips none
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) atomicMax(d.ztop_wr, d.nz - 1);
    using P = Sto<S>;
    __shared__ uint32_t slots[2][Q][BULK_THREADS];
    const int tid = threadIdx.x;
    const int x = blockIdx.x * BULK_THREADS + tid, y = blockIdx.y;
    const int z0 = blockIdx.z * LBMFS_BULK_PIPE_ZB, z1 = min(z0 + LBMFS_BULK_PIPE_ZB, d.nz);
    const bool in = x < d.nx;
    const bool xyin = x > 0 && x < d.nx - 1 && y > 0 && y < d.ny - 1;
    const long long sx = 1, sy = d.nx, sz = (long long)d.nx * d.ny;
    const long long irow = (long long)(in ? x : 0) + (long long)d.nx * y;
    auto flag_at = [&](int z) -> int { return (in && z < z1) ? (int)d.flags[irow + sz * z] : 0; };
    auto fast = [&](int fl, int z) -> bool { return fl == CL_L && xyin && z > 0 && z < d.nz - 1; };
    auto issue = [&](int z, int b) {
        const long long i = irow + sz * z;
#pragma unroll
        for (int q = 0; q < Q; ++q)
            cp_async4(&slots[b][q][tid], Pipe<S>::src(d, q, i - (cx(q) * sx + cy(q) * sy + cz(q) * sz)));
    };
    int fl_cur = flag_at(z0);
    bool fast_cur = fast(fl_cur, z0);
    if (fast_cur) issue(z0, 0);
    cp_async_commit();
    int fl_next = flag_at(z0 + 1);
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        const int b = (z - z0) & 1;
        const bool fast_next = z + 1 < z1 && fast(fl_next, z + 1);
        if (fast_next) issue(z + 1, b ^ 1);
        cp_async_commit();
        const int fl_after = flag_at(z + 2);
        const long long i = irow + sz * z;
        wl_append(d, (fl_cur & CL_MASK) == CL_I, WL_IFACE, (uint32_t)i);
        if (fast_cur) {
            cp_async_wait<1>();
            float fp[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q)
                fp[q] = Pipe<S>::get(&slots[b][0][tid], q, i - (cx(q) * sx + cy(q) * sy + cz(q) * sz), d.N);
            to_raw<S>(fp);
            collide_store<S>(d, fp, i);
        } else if (bulk_cell(fl_cur)) {
            liquid_one<S>(d, fl_cur, x, y, z, i);
        }
        fl_cur = fl_next;
        fl_next = fl_after;
        fast_cur = fast_next;
    }
    cp_async_wait<0>();
}

// ------------------------------------------------ staged bulk kernel (TMA)
//
// One block owns a row segment of BULK_THREADS cells at (y, z) for
// LBMFS_BULK_ZB consecutive z.  For every z it needs, per direction q, the
// source row (y - c_qy, z - c_qz) of plane q shifted by -c_qx: thread 0 stages
// those 19 rows (each widened by a 16-byte halo on both sides so that every
// copy starts 16-byte aligned) into shared memory with 1-D bulk copies that
// complete on an mbarrier, one z ahead of the rows being computed (double
// buffer).  Rows whose segment holds no interior liquid cell (gas, or the
// grid's boundary layers) are not staged.  Cells that need more than a plain
// pull (obstacle or wall neighbours) use the global-memory path.

template <int S> struct Stage;
template <> struct Stage<1> {  // float planes, halo 4 elements
    static constexpr int H = 4;
    static constexpr int ROW = BULK_THREADS + 2 * H;  // elements per staged row
    static constexpr int BYTES = Q * ROW * 4;
    static __device__ __forceinline__ const char *src(const Dev &d, int q, long long e) {
        return reinterpret_cast<const char *>(reinterpret_cast<const float *>(d.fsrc) + (long long)q * d.N + e);
    }
    static __device__ __forceinline__ int row_bytes(int) { return ROW * 4; }
    static __device__ __forceinline__ int row_off(int q) { return q * ROW * 4; }
    static __device__ __forceinline__ float get(const char *stage, int q, int k) {
        return reinterpret_cast<const float *>(stage + row_off(q))[k];
    }
};
template <> struct Stage<2> {  // q = 0 float (halo 4), q >= 1 half (halo 8)
    static constexpr int H0 = 4, H = 8;
    static constexpr int ROW0 = BULK_THREADS + 2 * H0, ROW = BULK_THREADS + 2 * H;
    static constexpr int BYTES = ROW0 * 4 + (Q - 1) * ROW * 2;
    static __device__ __forceinline__ const char *src(const Dev &d, int q, long long e) {
        if (q == 0) return reinterpret_cast<const char *>(reinterpret_cast<const float *>(d.fsrc) + e);
        const __half *hb = reinterpret_cast<const __half *>(reinterpret_cast<const float *>(d.fsrc) + d.N);
        return reinterpret_cast<const char *>(hb + (long long)(q - 1) * d.N + e);
    }
    static __device__ __forceinline__ int row_bytes(int q) { return q == 0 ? ROW0 * 4 : ROW * 2; }
    static __device__ __forceinline__ int row_off(int q) { return q == 0 ? 0 : ROW0 * 4 + (q - 1) * ROW * 2; }
    static __device__ __forceinline__ float get(const char *stage, int q, int k) {
        if (q == 0) return reinterpret_cast<const float *>(stage)[k];
        return __half2float(reinterpret_cast<const __half *>(stage + row_off(q))[k]) * F16_INV_SCALE;
    }
};


__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: gives up after ~2^22 polls (each try_wait also suspends for a
// hardware-chosen interval), far beyond any copy latency
constexpr int WAIT_POLLS = 1 << 22;
template <int POLLS = WAIT_POLLS> __device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity) {
    for (int it = 0; it < POLLS; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

template <int S>
__device__ __forceinline__ void stage_row(const Dev &d, char *stage, uint64_t *bar, int x0, int y, int z) {
    using G = Stage<S>;
    fence_async_shared();
    mbar_expect_tx(bar, G::BYTES);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        // the copy starts 16-byte aligned at x0 - h for every direction; the
        // x shift -c_qx is applied when the row is read
        int h = (S == 2 && q > 0) ? Stage<2>::H : 4;
        long long e = (long long)d.nx * ((y - cy(q)) + (long long)d.ny * (z - cz(q))) + x0 - h;
        bulk_g2s(stage + G::row_off(q), G::src(d, q, e), G::row_bytes(q), bar);
    }
}

template <int S>
__global__ void __launch_bounds__(BULK_THREADS, LBMFS_BULK_MINB) k_liquid_tma(Dev d) {
    // this variant visits every tile: record the grid's top so the next step skips none
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) atomicMax(d.ztop_wr, d.nz - 1);
    using P = Sto<S>;
    using G = Stage<S>;
    extern __shared__ __align__(128) char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);  // two mbarriers
    char *buf0 = smem + 128;
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * BULK_THREADS, x = x0 + tid, y = blockIdx.y;
    const int z0 = blockIdx.z * LBMFS_BULK_ZB, z1 = min(z0 + LBMFS_BULK_ZB, d.nz);
    const bool in = x < d.nx;
    const bool xin = x > 0 && x < d.nx - 1;
    const bool yin = y > 0 && y < d.ny - 1;
    bool failed = false;
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    unsigned phase[2] = {0u, 0u};
    auto flag_at = [&](int z) -> int {
        return (in && z < z1) ? (int)d.flags[x + (long long)d.nx * (y + (long long)d.ny * z)] : 0;
    };
    auto fast = [&](int fl, int z) -> bool { return fl == CL_L && xin && yin && z > 0 && z < d.nz - 1; };
    int fl_cur = flag_at(z0);
    bool staged_cur = __syncthreads_or(fast(fl_cur, z0)) != 0;
    if (staged_cur && tid == 0) stage_row<S>(d, buf0, &bar[0], x0, y, z0);
    int fl_next = flag_at(z0 + 1);
    for (int z = z0; z < z1; ++z) {
        const int b = (z - z0) & 1;
        char *stage = buf0 + b * G::BYTES;
        // every thread is done with the other buffer (previous row) here
        bool staged_next = __syncthreads_or(z + 1 < z1 && fast(fl_next, z + 1)) != 0;
        if (staged_next && tid == 0) stage_row<S>(d, buf0 + (b ^ 1) * G::BYTES, &bar[b ^ 1], x0, y, z + 1);
        int fl_after = flag_at(z + 2);
        const long long i = (long long)(in ? x : 0) + (long long)d.nx * (y + (long long)d.ny * z);
        const int c = fl_cur;
        wl_append(d, (c & CL_MASK) == CL_I, WL_IFACE, (uint32_t)i);
        if (staged_cur) {
            // every thread keeps stepping through the block barriers even if
            // its wait gives up; the outcome is settled after the loop
            if (!mbar_wait(&bar[b], phase[b])) failed = true;
            phase[b] ^= 1u;
        }
        if (fast(c, z)) {
            float fp[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) fp[q] = G::get(stage, q, tid + ((S == 2 && q > 0) ? Stage<2>::H : 4) - cx(q));
            to_raw<S>(fp);
            collide_store<S>(d, fp, i);
        } else if (bulk_cell(c)) {
            liquid_one<S>(d, c, x, y, z, i);
        }
        fl_cur = fl_next;
        fl_next = fl_after;
        staged_cur = staged_next;
    }
    if (__syncthreads_or(failed)) {
        // a staged copy did not complete in time: report it; every staged row
        // has had its (bounded) wait above, so no copy is left unawaited
        if (tid == 0) atomicOr(d.status, ST_TIMEOUT);
    }
}

// --------------------------------------------------- ring bulk kernel
//
// The bulk kernel of the FP16 storage.  Pull streaming reads population q of
// cell i at i - (c_x + c_y nx + c_z nx ny): a shift of the linear cell index, so
// the sources of TILE consecutive cells are TILE consecutive elements of each
// plane whatever the grid's sizes, and 19 linear bulk copies (1 KB each) bring a
// tile's arriving populations into shared memory.  A producer warp keeps a ring
// of STAGES tiles in flight per block with no registers held for them, which
// was what bound the one-cell-per-thread kernel (64 registers, 24 warps with one
// cell's loads each; FP16S: 73 % of the issue slots, 52 % of the copy
// bandwidth); the consumer warps take two cells per thread, in packed FP32
// arithmetic with half the instructions per cell.  Copies start at the 16-byte
// boundary below the source; the remainder m_q depends on q only (tiles start
// at multiples of TILE).  Reads past a plane's ends meet the next plane or the
// guard bands and belong to cells on grid faces, whose populations from beyond
// the face are their own (resting walls) or a periodic image's.  On the x faces
// -- two cells of every row, so some in nearly every warp -- a second warp
// fetches them as soon as a tile is announced and patches them into the staged
// tile; the consumers fetch those of the y and z faces (whole warps) themselves.
// Fetching the x faces in the consumers too cost a global load's latency per
// warp: 768x384x256 bulk kernel 763 us against 581 without any face work.
// Measured, us, before (one cell per thread) and now: 768x384x256 856 and 593
// (5.1 TB/s, 76 % of the copy bandwidth; on 384x192x128 issue is 59 % and the FMA
// pipe 47 % active, so no unit alone is the bound),
// 385x190x127 127 and 91, 64 tanks of edge 48..112 626 and 408.  On grids too
// small to fill the GPU it is even (130x40x40 11 and 12).  The FP32 storage
// keeps the other kernel: 944 us against 1021 in a ring, HBM-bound either way.
constexpr int RING_STAGES = 4;
struct RingShape {
    static constexpr int TILE = RING_TILE, ESZ = 2;         // cells, bytes per moving population
    static constexpr int WORKERS = TILE / 2, THREADS = WORKERS + 64;  // and the producer and the patching warp
    static constexpr int ALIGN = 16 / ESZ;                  // elements per 16 bytes
    static constexpr int ROW = (TILE + ALIGN) * ESZ;        // bytes of one staged plane, q >= 1
    static constexpr int COPY = TILE * 4 + (Q - 1) * ROW;   // bytes of a tile's copies
    static constexpr int STAGE = (COPY + TILE + 127) / 128 * 128;  // populations, then the flags
    static constexpr int HEAD = 256;                        // barriers, tile descriptors
    static constexpr int SMEM = HEAD + RING_STAGES * STAGE;
};
// offset of direction q's source in the linear cell index
__device__ __forceinline__ int src_offset(const Dev &d, int q) { return cx(q) + d.nx * (cy(q) + d.ny * cz(q)); }
// element index, from the grid's (16-byte aligned) start, of the first staged
// element of plane q >= 1 for the tile at i0, before the rounding to 16 bytes
// (the FP16 planes start after plane 0, whose N floats are 2 N of their
// elements)
__device__ __forceinline__ long long ring_plane(const Dev &d, int q) { return (long long)(q + 1) * d.N; }

// what a tile is: its tank (batch) and first cell; tank < 0 ends the ring
struct RingTile {
    int tank;
    uint32_t i0;
};

// The populations of the cells 2p, 2p + 1 of the staged tile in raw units.
// EVEN (nx and the cell count even): a pair starts on an even element exactly
// when c_x = 0; else that is decided per direction at run time.
template <bool EVEN>
__device__ __forceinline__ float2 ring_pair(const char *stage, const Dev &d, int q, int p) {
    using G = RingShape;
    if (q == 0) return *reinterpret_cast<const float2 *>(stage + 8 * p);
    const int m = (int)(ring_plane(d, q) - src_offset(d, q)) & (G::ALIGN - 1);  // (tiles start at multiples of ALIGN)
    const uint32_t *w = reinterpret_cast<const uint32_t *>(stage + G::TILE * 4 + (q - 1) * G::ROW) + p + (m >> 1);
    uint32_t v;
    if (EVEN && cx(q) == 0) v = w[0];
    else v = __funnelshift_r(w[0], w[1], EVEN ? 16 : (m & 1) * 16);
    return __half22float2(*reinterpret_cast<const __half2 *>(&v));
}
// the five directions with component `sign` along an axis, 5 bits each
__host__ __device__ constexpr unsigned face_dirs(int axis, int sign) {
    unsigned b = 0;
    int n = 0;
    for (int q = 1; q < Q; ++q)
        if ((axis == 0 ? cx(q) : (axis == 1 ? cy(q) : cz(q))) == sign) b |= (unsigned)q << (5 * n++);
    return b;
}
// Where the population that arrives at face cell i from beyond the grid in
// direction q is read: the cell's own opposite one (resting wall) or the
// periodic image's, as an element index.
__device__ __forceinline__ long long face_source(const Dev &d, uint32_t i, int q) {
    if (d.periodic) {
        int x, y, z;
        coords(d, i, x, y, z);
        const long long si = nbr(d, x, y, z, -dir_x(q), -dir_y(q), -dir_z(q));
        if (si >= 0) return ring_plane(d, q) + si;
    }
    return ring_plane(d, opp_lane(q)) + i;
}
// byte offset in a stage of population q of the tile's cell `local`
__device__ __forceinline__ int stage_slot(const Dev &d, int q, int local) {
    using G = RingShape;
    const int off = dir_x(q) + d.nx * (dir_y(q) + d.ny * dir_z(q));
    const int m = (int)(ring_plane(d, q) - off) & (G::ALIGN - 1);
    return G::TILE * 4 + (q - 1) * G::ROW + (local + m) * G::ESZ;
}
// A cell on a y or z face, by the consumer that owns it: its populations from
// beyond the face into its own slots of the staged tile.  (A loop over the two
// axes and five directions each: the code stays small.)
__device__ __forceinline__ void ring_face(const Dev &d, char *stage, uint32_t i, int local) {
    const uint16_t *src = reinterpret_cast<const uint16_t *>(d.fsrc);
    int x, y, z;
    coords(d, i, x, y, z);
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {  // y low, y high, z low, z high
        const int p = s < 2 ? y : z, end = (s < 2 ? d.ny : d.nz) - 1;
        if (p != (s & 1 ? end : 0)) continue;
        const unsigned dirs = s < 2 ? (s & 1 ? face_dirs(1, -1) : face_dirs(1, 1)) : (s & 1 ? face_dirs(2, -1) : face_dirs(2, 1));
        uint16_t v[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = __ldg(src + face_source(d, i, (int)(dirs >> (5 * j) & 31u)));
#pragma unroll
        for (int j = 0; j < 5; ++j)
            *reinterpret_cast<uint16_t *>(stage + stage_slot(d, (int)(dirs >> (5 * j) & 31u), local)) = v[j];
    }
}
// The patching warp's work on one tile: per row boundary b inside it, the five
// directions with c_x > 0 of cell b (x = 0) and the five with c_x < 0 of cell
// b - 1 (x = nx - 1).  A lane keeps one of the ten (three rows at a time), so
// that an item is an addition, a load and a 2-byte store.  The loads of a tile
// are issued before the previous tile's are stored.
struct RingPatch {
    static constexpr int U = 4;  // items per lane held at a time: 12 rows, enough for one round from nx = 47 up
    uint16_t v[U];
    int at[U];  // byte offset of the slot in the stage, -1: none
    uint32_t rows, row0, i0;
    // boundaries b = row nx with i0 <= b <= i0 + TILE
    __device__ __forceinline__ void begin(const Dev &d, uint32_t first) {
        const uint32_t nx = (uint32_t)d.nx;
        i0 = first;
        row0 = (i0 + nx - 1) / nx;
        rows = (i0 + RingShape::TILE) / nx + 1 - row0;
    }
    __device__ __forceinline__ void load(const Dev &d, uint32_t r0) {
        const uint32_t lane = threadIdx.x & 31u, j = lane % 10u;
        const bool high = j >= 5;
        const int q = (int)((high ? face_dirs(0, -1) >> (5 * (j - 5u)) : face_dirs(0, 1) >> (5 * j)) & 31u);
        const uint16_t *own = reinterpret_cast<const uint16_t *>(d.fsrc) + ring_plane(d, opp_lane(q));
        const int slot = stage_slot(d, q, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t r = r0 + 3u * u + lane / 10u;
            const uint32_t i = (row0 + r) * (uint32_t)d.nx - (high ? 1u : 0u);  // (of b = i0: before the tile)
            at[u] = -1;
            if (lane < 30 && r < rows && i >= i0 && i < i0 + RingShape::TILE && i < (uint32_t)d.N) {
                v[u] = __ldg(d.periodic ? reinterpret_cast<const uint16_t *>(d.fsrc) + face_source(d, i, q) : own + i);
                at[u] = slot + (int)(i - i0) * RingShape::ESZ;
            }
        }
    }
    __device__ __forceinline__ void store(char *stage) const {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (at[u] >= 0) *reinterpret_cast<uint16_t *>(stage + at[u]) = v[u];
    }
};

// One staged tile by the consumer warps.  The kernel holds one copy of the
// collision (with one per parity and per kind of store its instructions did not
// fit the caches: 4.7 of 14 stall cycles per instruction in a batch): the
// gather and the stores branch on the tank's parity, and the collided pairs are
// kept packed, a register per direction, until the stores.
template <bool ZG>
__device__ __forceinline__ void ring_tile(const Dev &d, char *stage, uint64_t *empty, uint32_t i0, int p) {
    using G = RingShape;
    const unsigned cc = *reinterpret_cast<const uint16_t *>(stage + G::COPY + 2 * p);
    const int c0 = (int)(cc & 0xffu), c1 = (int)(cc >> 8);
    const int lane = threadIdx.x & 31;
    const uint32_t i = i0 + 2u * (uint32_t)p;
    // interface cells are listed, in cell order
    const bool f0 = (c0 & CL_MASK) == CL_I, f1 = (c1 & CL_MASK) == CL_I;
    const unsigned m0 = __ballot_sync(0xffffffffu, f0), m1 = __ballot_sync(0xffffffffu, f1);
    if (m0 | m1) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&d.cnt[WL_IFACE], (uint32_t)(__popc(m0) + __popc(m1)));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m0 & ((1u << lane) - 1u)) + __popc(m1 & ((1u << lane) - 1u));
        // (repeated launches on one state, as the batch's autotuner does them,
        // append again)
        if (at + 2 <= d.cap || at + (f0 ? 1 : 0) + (f1 ? 1 : 0) <= d.cap) {
            if (f0) d.list[WL_IFACE][at++] = i;
            if (f1) d.list[WL_IFACE][at] = i + 1;
        } else {
            atomicOr(d.status, ST_OVERFLOW);
        }
    }
    const bool s0 = bulk_cell(c0), s1 = bulk_cell(c1);
    if (!__any_sync(0xffffffffu, s0 || s1)) {
        if (lane == 0) mbar_arrive(empty);
        return;
    }
    if ((s0 && (c0 & FACE_YZ)) || (s1 && (c1 & FACE_YZ))) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h)
            if (h ? s1 && (c1 & FACE_YZ) : s0 && (c0 & FACE_YZ)) ring_face(d, stage, i + h, 2 * p + h);
    }
    float2 fp[Q];
    if (d.pair_ok) {
#pragma unroll
        for (int q = 0; q < Q; ++q) fp[q] = ring_pair<true>(stage, d, q, p);
    } else {
#pragma unroll
        for (int q = 0; q < Q; ++q) fp[q] = ring_pair<false>(stage, d, q, p);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty);  // the stage is in registers
    if (!(s0 || s1)) return;
    float2 rest;
    uint32_t hp[Q];  // the collided pairs as stored
    const float2 rho = collide_store_v<Sto<2>::SCALE, ZG, float2>(d, fp, [&](int q, float2 v) {
        if (q == 0) {
            rest = v;
            return v;
        }
        const __half2 h = __floats2half2_rn(v.x, v.y);
        hp[q] = *reinterpret_cast<const uint32_t *>(&h);
        return __half22float2(h);
    });
    float *w0 = reinterpret_cast<float *>(d.fdst) + i;
    const bool both = s0 && s1;
    if (__all_sync(__activemask(), both) && d.pair_ok) {
        *reinterpret_cast<float2 *>(w0) = rest;
#pragma unroll
        for (int q = 1; q < Q; ++q)
            *reinterpret_cast<uint32_t *>(reinterpret_cast<uint16_t *>(d.fdst) + ring_plane(d, q) + i) = hp[q];
    } else {
        // some pair has a cell that is not stepped here, or an odd cell count
        // puts every other plane on an odd element
        const bool skew = d.N & 1;
        if (s0) w0[0] = rest.x;
        if (s1) w0[1] = rest.y;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            uint16_t *w = reinterpret_cast<uint16_t *>(d.fdst) + ring_plane(d, q) + i;
            const bool word = both && !(q % 2 == 0 && skew);
            if (word) *reinterpret_cast<uint32_t *>(w) = hp[q];
            if (s0 && !word) w[0] = (uint16_t)hp[q];
            if (s1 && !word) w[1] = (uint16_t)(hp[q] >> 16);
        }
    }
    if ((s0 && !vpos_finite(rho.x)) || (s1 && !vpos_finite(rho.y))) atomicOr(d.status, ST_NONFINITE);
}

// The ring over a launch's n entries: tile_of(entry) gives an entry's tank and
// first cell (single tank: tank 0), dev_of(tank) its descriptor.  Warps 0 .. are
// the consumers, then the producer, then the patching warp.  A stage goes
// through four barriers: announced (its tile and class bytes are written),
// landed (its copies are complete), full (patched), empty (in registers).
// Every wait is bounded (ring_wait); one that gives up ends its warp's role, and
// the others' by their own waits.  The block then waits for its copies in
// flight and sets the sticky status of every tank that it had tiles of: any of
// them may hold cells that were not stepped.
#ifndef LBMFS_RING_POLLS
#define LBMFS_RING_POLLS WAIT_POLLS  // polls of a role's wait (0: a test's waits that all give up)
#endif
__device__ __forceinline__ bool ring_wait(uint64_t *bar, unsigned parity) {
    return __all_sync(0xffffffffu, mbar_wait<LBMFS_RING_POLLS>(bar, parity));
}
template <bool ZG, class TileOf, class DevOf>
__device__ __forceinline__ void ring_run(uint32_t n, TileOf tile_of, DevOf dev_of) {
    using G = RingShape;
    extern __shared__ __align__(128) char smem[];
    uint64_t *said = reinterpret_cast<uint64_t *>(smem), *landed = said + RING_STAGES, *full = landed + RING_STAGES,
             *empty = full + RING_STAGES;
    RingTile *desc = reinterpret_cast<RingTile *>(empty + RING_STAGES);
    static_assert(RING_STAGES * (4 * 8 + sizeof(RingTile)) <= G::HEAD, "barriers and descriptors fit the head");
    char *stages = smem + G::HEAD;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        for (int k = 0; k < RING_STAGES; ++k) {
            mbar_init(&said[k], 1);
            mbar_init(&landed[k], 1);
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], G::WORKERS / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    bool ok = true;
    uint32_t made = 0;  // tiles produced
    if (tid < G::WORKERS) {
        for (uint32_t k = 0;; ++k) {
            const int st = (int)(k % RING_STAGES);
            const unsigned ph = (k / RING_STAGES) & 1u;
            ok = ring_wait(&full[st], ph) && ring_wait(&landed[st], ph);
            if (!ok) break;
            const RingTile t = desc[st];
            if (t.tank < 0) break;
            ring_tile<ZG>(dev_of(t.tank), stages + st * G::STAGE, &empty[st], t.i0, tid);
        }
    } else if (tid < G::WORKERS + 32) {
        uint32_t &k = made;
        int top_tank = -1, top = -1;  // highest plane with fluid of the current tank's tiles
        auto flush_top = [&]() {
            if (lane == 0 && top >= 0) atomicMax(dev_of(top_tank).ztop_wr, top);
        };
        for (uint32_t base = blockIdx.x; base < n && ok; base += 32u * gridDim.x) {
            // a lane per entry: tiles above the previous step's fluid (plus a
            // margin) hold only gas
            const uint32_t e = base + (uint32_t)lane * gridDim.x;
            RingTile t{-1, 0};
            if (e < n) {
                t = tile_of(e);
                const Dev &d = dev_of(t.tank);
                if ((int)(t.i0 / ((uint32_t)d.nx * (uint32_t)d.ny)) > __ldg(d.ztop_rd) + ZTOP_MARGIN) t.tank = -1;
            }
            // the class bytes of the next tile are requested before the current
            // one waits for a free stage (the flags are padded to whole tiles)
            unsigned todo = __ballot_sync(0xffffffffu, t.tank >= 0);
            auto fetch = [&](unsigned rest, int &tank, uint32_t &i0) {
                const int l = rest ? __ffs(rest) - 1 : 0;
                tank = __shfl_sync(0xffffffffu, t.tank, l);
                i0 = __shfl_sync(0xffffffffu, t.i0, l);
                uint4 f = make_uint4(0, 0, 0, 0);
                if (rest) {
                    const char *src = reinterpret_cast<const char *>(dev_of(tank).flags) + i0;
                    static_assert(G::TILE == 512, "16 class bytes per lane");
                    f = reinterpret_cast<const uint4 *>(src)[lane];
                }
                return f;
            };
            int tank;
            uint32_t i0;
            uint4 fl = fetch(todo, tank, i0);
            while (todo && ok) {
                todo &= todo - 1;
                int tank1;
                uint32_t i1;
                const uint4 fl1 = fetch(todo, tank1, i1);
                const Dev &d = dev_of(tank);
                const unsigned any = fl.x | fl.y | fl.z | fl.w;
                const bool any_wet = __any_sync(0xffffffffu, (any & 0x03030303u) != 0),
                           any_liq = __any_sync(0xffffffffu, (any & 0x01010101u) != 0);
                if (any_wet) {
                    const int st = (int)(k % RING_STAGES);
                    char *stage = stages + st * G::STAGE;
                    if (tank != top_tank) {
                        flush_top();
                        top_tank = tank;
                        top = -1;
                    }
                    top = max(top, min(d.nz - 1, (int)((i0 + G::TILE - 1) / ((uint32_t)d.nx * (uint32_t)d.ny))));
                    if (k >= RING_STAGES) ok = ring_wait(&empty[st], (k / RING_STAGES - 1) & 1u);
                    if (!ok) break;
                    reinterpret_cast<uint4 *>(stage + G::COPY)[lane] = fl;
                    if (lane == 0) desc[st] = RingTile{tank, i0};
                    fence_async_shared();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&said[st]);
                        mbar_expect_tx(&landed[st], any_liq ? (unsigned)G::COPY : 0u);
                    }
                    __syncwarp();
                    if (any_liq && lane < Q) {
                        if (lane == 0) {
                            bulk_g2s(stage, reinterpret_cast<const float *>(d.fsrc) + i0, G::TILE * 4, &landed[st]);
                        } else {
                            const int off = dir_x(lane) + d.nx * (dir_y(lane) + d.ny * dir_z(lane));
                            const long long first = ring_plane(d, lane) + i0 - off;
                            bulk_g2s(stage + G::TILE * 4 + (lane - 1) * G::ROW,
                                     reinterpret_cast<const char *>(d.fsrc) + (first & ~(long long)(G::ALIGN - 1)) * G::ESZ,
                                     G::ROW, &landed[st]);
                        }
                    }
                    ++k;
                }
                tank = tank1;
                i0 = i1;
                fl = fl1;
            }
        }
        flush_top();
        const int st = (int)(k % RING_STAGES);
        if (ok && k >= RING_STAGES) ok = ring_wait(&empty[st], (k / RING_STAGES - 1) & 1u);
        if (ok && lane == 0) {
            desc[st] = RingTile{-1, 0};
            mbar_arrive(&said[st]);
            mbar_expect_tx(&landed[st], 0u);
        }
    } else {
        // tile k is patched while tile k + 1's loads, where it is announced
        // already, are under way
        RingPatch cur, next;
        auto stage_of = [&](uint32_t k) { return (int)(k % RING_STAGES); };
        auto phase_of = [&](uint32_t k) { return (k / RING_STAGES) & 1u; };
        auto begin = [&](RingPatch &r, uint32_t k) {  // after tile k's announcement; its tank
            const RingTile t = desc[stage_of(k)];
            if (t.tank >= 0) {
                r.begin(dev_of(t.tank), t.i0);
                if (r.rows) r.load(dev_of(t.tank), 0);
            }
            return t.tank;
        };
        ok = ring_wait(&said[0], 0);
        int tank = ok ? begin(cur, 0) : -1;
        for (uint32_t k = 0; ok; ++k) {
            const int st = stage_of(k);
            int tank1 = -1;
            const bool more = tank >= 0;
            const bool ready = more && __all_sync(0xffffffffu, mbar_try_wait(&said[stage_of(k + 1)], phase_of(k + 1)));
            if (ready) tank1 = begin(next, k + 1);
            if (more && cur.rows) {
                ok = ring_wait(&landed[st], phase_of(k));
                char *stage = stages + st * G::STAGE;
                cur.store(stage);
                for (uint32_t r0 = 3u * RingPatch::U; r0 < cur.rows; r0 += 3u * RingPatch::U) {
                    cur.load(dev_of(tank), r0);
                    cur.store(stage);
                }
                __syncwarp();
            }
            if (lane == 0) mbar_arrive(&full[st]);
            if (!more || !ok) break;
            if (!ready) {
                ok = ring_wait(&said[stage_of(k + 1)], phase_of(k + 1));
                tank1 = ok ? begin(next, k + 1) : -1;
            }
            cur = next;
            tank = tank1;
        }
    }
    if (__syncthreads_or(!ok)) {
        if (tid >= G::WORKERS && tid < G::WORKERS + 32)
            for (uint32_t k = made > RING_STAGES ? made - RING_STAGES : 0; k < made; ++k)
                mbar_wait(&landed[k % RING_STAGES], (k / RING_STAGES) & 1u);
        for (uint32_t e = blockIdx.x + (uint32_t)tid * gridDim.x; e < n; e += G::THREADS * gridDim.x)
            atomicOr(dev_of(tile_of(e).tank).status, ST_TIMEOUT);
    }
}
struct OneTank {
    const Dev &d;
    __device__ __forceinline__ const Dev &operator()(int) const { return d; }
};
struct ManyTanks {
    const TankSet &ts;
    __device__ __forceinline__ const Dev &operator()(int tank) const { return ts.d[tank]; }
};
template <bool ZG>
__global__ void __launch_bounds__(RingShape::THREADS, RING_CTAS) k_ring(const __grid_constant__ Dev d, uint32_t n) {
    ring_run<ZG>(n, [](uint32_t e) { return RingTile{0, e * (uint32_t)RingShape::TILE}; }, OneTank{d});
}

// the ring over all tanks of a batch's launch (entries: tank, tile in x + 2^16 y)
template <bool ZG>
__global__ void __launch_bounds__(RingShape::THREADS, RING_CTAS)
    k_batch_ring(const __grid_constant__ TankSet ts, const Tile *__restrict__ table, unsigned n) {
    ring_run<ZG>(n,
                         [&](uint32_t e) {
                             const Tile t = table[e];
                             return RingTile{t.tank, (t.x + ((uint32_t)t.y << 16)) * (uint32_t)RingShape::TILE};
                         },
                         ManyTanks{ts});
}

// fill level of a neighbour as seen by the normal estimate
__device__ __forceinline__ double fill_seen(const Dev &d, long long ni, double own) {
    int c = cls(d, ni);
    if (c == CL_L) return 1.0;
    if (c == CL_I) return d.phisrc[ni];
    if (c == CL_G) return 0.0;
    return own;
}

// ---- Sec. 2.2 Laplace pressure: mean curvature kappa = div(n^)/2 at an
// interface cell from the unit normals of its six axis neighbours (central
// differences; the normals are those of the reconstruction, -grad(phi) with
// the same fill-level rules); an obstacle or wall neighbour takes the cell's
// own unit normal nc.  A liquid sphere of radius R has kappa = 1/R.
__device__ __forceinline__ void unit_vec_d(const double *n, double *out) {
    double len = sqrt((n[0] * n[0] + n[1] * n[1]) + n[2] * n[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) out[k] = len > 0.0 ? n[k] / len : 0.0;
}
__device__ __noinline__ double curvature_d(const Dev &d, int x, int y, int z, double nc0, double nc1, double nc2) {
    const double nc[3] = {nc0, nc1, nc2};
    double div = 0.0;
    for (int k = 0; k < 3; ++k) {
        double comp[2];
        for (int sgn = 0; sgn < 2; ++sgn) {
            const int s = sgn ? -1 : 1;
            const long long yi = nbr(d, x, y, z, k == 0 ? s : 0, k == 1 ? s : 0, k == 2 ? s : 0);
            const int c = cls(d, yi);
            if (c == CL_WALL || c == CL_O) {
                comp[sgn] = nc[k];
                continue;
            }
            int yx, yy, yz;
            coords(d, yi, yx, yy, yz);
            const double own = c == CL_L ? 1.0 : (c == CL_I ? d.phisrc[yi] : 0.0);
            double n[3], nh[3];
            for (int j = 0; j < 3; ++j) {
                const double pm = fill_seen(d, nbr(d, yx, yy, yz, j == 0 ? -1 : 0, j == 1 ? -1 : 0, j == 2 ? -1 : 0), own);
                const double pp = fill_seen(d, nbr(d, yx, yy, yz, j == 0 ? 1 : 0, j == 1 ? 1 : 0, j == 2 ? 1 : 0), own);
                n[j] = 0.5 * (pm - pp);
            }
            unit_vec_d(n, nh);
            comp[sgn] = nh[k];
        }
        div += comp[0] - comp[1];
    }
    return 0.25 * div;
}
// The same in float for the float storages, one axis: member r of a cell's trio
// takes the two neighbours on axis r, own the cell's unit normal's component r;
// the caller adds the three in axis order.  All classes and fill levels around
// the two neighbours are requested at once (one thread walking the six
// neighbours' six neighbours class by class was most of the interface kernel:
// 64^3 bubble 20 us).
__device__ __noinline__ float curvature_axis_f(const Dev &d, int x, int y, int z, int r, float own) {
    const int ex = r == 0, ey = r == 1, ez = r == 2;
    float comp[2], f[2][6];
    int cy0[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int sg = s ? -1 : 1;
        const long long yi = nbr(d, x, y, z, sg * ex, sg * ey, sg * ez);
        cy0[s] = cls(d, yi);
        int yx = x, yy = y, yz = z;
        if (yi >= 0) coords(d, yi, yx, yy, yz);
        const long long at = yi >= 0 ? yi : x + (long long)d.nx * (y + (long long)d.ny * z);
        const float ph = d.phifsrc[at];
        const float self = cy0[s] == CL_L ? 1.0f : (cy0[s] == CL_I ? ph : 0.0f);
        int c[6];
        float p[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int sj = j & 1 ? 1 : -1;
            const long long ni = nbr(d, yx, yy, yz, j < 2 ? sj : 0, j >= 2 && j < 4 ? sj : 0, j >= 4 ? sj : 0);
            c[j] = cls(d, ni);
            p[j] = d.phifsrc[ni < 0 ? at : ni];
        }
#pragma unroll
        for (int j = 0; j < 6; ++j)
            f[s][j] = c[j] == CL_L ? 1.0f : (c[j] == CL_I ? p[j] : (c[j] == CL_G ? 0.0f : self));
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const float n0 = 0.5f * (f[s][0] - f[s][1]), n1 = 0.5f * (f[s][2] - f[s][3]), n2 = 0.5f * (f[s][4] - f[s][5]);
        const float len = sqrtf((n0 * n0 + n1 * n1) + n2 * n2);
        const float nr = r == 0 ? n0 : (r == 1 ? n1 : n2);
        comp[s] = (cy0[s] == CL_WALL || cy0[s] == CL_O) ? own : (len > 0.0f ? nr / len : 0.0f);
    }
    return comp[0] - comp[1];
}

// ---- C1 + C2 for interface cells of the float storages: three threads per
// cell.  Member r of a cell's trio owns three pairs of opposite directions
// (r = 0: W/E, TW/BE, TE/BW; r = 1: N/S, TN/BS, TS/BN; r = 2: T/B, NW/SE,
// NE/SW), so the bounce-back, reconstruction and mass exchange of a link,
// which pair q with qbar, stay inside one thread, and the first pair of
// member r is the axis pair of component r of the normal.  Sums over all
// directions (density, momentum, exchanged mass, the stored cell sum) are
// formed per member and added as member 0 + member 1 + member 2 on all three
// threads, so a trio agrees bit for bit.  Ten trios per warp; lanes 30 and 31
// shadow the last trio and write nothing.
//
// A double operation holds a scheduler for 64 cycles (a conversion about 100,
// a division 550), whatever the number of active lanes: they bound this kernel
// when each trio converted the fill levels it read and did its own mass update
// (about 1800 of those cycles per 10 cells).  The fill levels are therefore
// also kept rounded to float, and a warp takes 30 cells as `sub` = 3 rounds of
// ten trios before lane l does the mass update of cell l for all of them; a
// list too short to give every scheduler a warp that way takes ten cells per
// warp (sub = 1).  64-tank FP16S batch 154 us with sub = 1, 137 with 3; alone on
// 768x384x256 102 and 116, beside the bulk kernel the step is the same.

// neighbour (x + dx, y + dy, z + dz) as a 32-bit cell index without
// branches (periodic axes wrap); -1 beyond a wall
__device__ __forceinline__ int nbr32(const Dev &d, int x, int y, int z, int dx, int dy, int dz) {
    int px = x + dx, py = y + dy, pz = z + dz;
    const bool ox = px < 0 || px >= d.nx, oy = py < 0 || py >= d.ny, oz = pz < 0 || pz >= d.nz;
    px = px < 0 ? px + d.nx : (px >= d.nx ? px - d.nx : px);
    py = py < 0 ? py + d.ny : (py >= d.ny ? py - d.ny : py);
    pz = pz < 0 ? pz + d.nz : (pz >= d.nz ? pz - d.nz : pz);
    const bool wall = (ox && !(d.periodic & 1u)) || (oy && !(d.periodic & 2u)) || (oz && !(d.periodic & 4u));
    return wall ? -1 : px + d.nx * (py + d.ny * pz);
}
// moving population q >= 1 of cell j as a float deviation (no branch on q)
template <int S> __device__ __forceinline__ float trio_ld(const void *g, int q, uint32_t j, long long N) {
    if constexpr (S == 1) return __ldg(reinterpret_cast<const float *>(g) + ((long long)q * N + j));
    else return __half2float(__ldg(Sto<2>::hp(g, N) + ((long long)(q - 1) * N + j))) * F16_INV_SCALE;
}
// store moving population q >= 1 of cell j; returns the value as stored
template <int S> __device__ __forceinline__ float trio_st(void *g, int q, uint32_t j, long long N, float v) {
    if constexpr (S == 1) {
        pop_st(reinterpret_cast<float *>(g) + ((long long)q * N + j), v);
        return v;
    } else {
        const __half h = __float2half_rn(v * F16_SCALE);
        pop_st(const_cast<__half *>(Sto<2>::hp(g, N)) + ((long long)(q - 1) * N + j), h);
        return __half2float(h) * F16_INV_SCALE;
    }
}
__host__ __device__ constexpr int trio_q(int r, int k) {
    return r == 0 ? (k == 0 ? 1 : (k == 1 ? 7 : 8)) : (r == 1 ? (k == 0 ? 3 : (k == 1 ? 9 : 10)) : (k == 0 ? 5 : (k == 1 ? 11 : 12)));
}
__host__ __device__ constexpr bool trio_ok() {
    int seen = 0;
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) {
            const int q = trio_q(r, k), b = opp(q);
            if ((seen >> q) & 1 || (seen >> b) & 1) return false;
            seen |= (1 << q) | (1 << b);
            if ((k == 0) != (q <= 6)) return false;  // the first pair is the axis pair
        }
    return seen == (1 << Q) - 2 && trio_q(0, 0) == 1 && trio_q(1, 0) == 3 && trio_q(2, 0) == 5;
}
static_assert(trio_ok(), "trio pairs: each moving direction once, axis pair first");
// the value f(q) for the first direction q of pair k of member r (three
// compile-time constants, selected by r)
template <int K, class F> __device__ __forceinline__ int trio_sel(int r, F f) {
    return r == 0 ? f(trio_q(0, K)) : (r == 1 ? f(trio_q(1, K)) : f(trio_q(2, K)));
}
__device__ __forceinline__ float trio_sum(float v, int b3) {
    const float a = __shfl_sync(0xffffffffu, v, b3), b = __shfl_sync(0xffffffffu, v, b3 + 1),
                c = __shfl_sync(0xffffffffu, v, b3 + 2);
    return (a + b) + c;
}
// f_eq(rho_g, u) - w for a direction of weight w with c.u = cu
__device__ __forceinline__ float feq_dev_cu(float w, float cu, float usq, float drg) {
    const float s = 3.0f * cu + 4.5f * cu * cu - 1.5f * usq;
    return w * (drg + s + drg * s);
}

template <int S>
__device__ __forceinline__ void interface_trio(const Dev &d, const VB &vb) {
    using P = Sto<S>;
    const long long N = d.N;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool lane_ok = lane < 30;
    const int g = lane_ok ? lane / 3 : 9;             // trio of the warp
    const int r = lane_ok ? lane - 3 * g : lane - 30;  // member
    const int b3 = 3 * g;
    // pair k: first direction a = trio_q(r, k) with velocity e, second b = opp(a)
    // with -e; sg = +1 when a is the pair member whose leading nonzero
    // component is positive (the collision's split, see collide_store_v).
    // Packed in one word per pair (a, b: 5 bits each; e + 1: 2 bits per
    // component; sg > 0: 1 bit) to keep the loop's registers for the cells.
    uint32_t pk[3];
    const auto pack = [](int q) {
        const bool pos = cx(q) > 0 || (cx(q) == 0 && (cy(q) > 0 || (cy(q) == 0 && cz(q) > 0)));
        return q | (opp(q) << 5) | ((cx(q) + 1) << 10) | ((cy(q) + 1) << 12) | ((cz(q) + 1) << 14) | ((pos ? 1 : 0) << 16);
    };
    pk[0] = (uint32_t)trio_sel<0>(r, pack);
    pk[1] = (uint32_t)trio_sel<1>(r, pack);
    pk[2] = (uint32_t)trio_sel<2>(r, pack);
#define TRIO_QA(k) ((int)(pk[k] & 31u))
#define TRIO_QB(k) ((int)((pk[k] >> 5) & 31u))
#define TRIO_EX(k) ((int)((pk[k] >> 10) & 3u) - 1)
#define TRIO_EY(k) ((int)((pk[k] >> 12) & 3u) - 1)
#define TRIO_EZ(k) ((int)((pk[k] >> 14) & 3u) - 1)
#define TRIO_POS(k) ((pk[k] >> 16) & 1u)
    const float ax = d.a_f[0], ay = d.a_f[1], az = d.a_f[2];
    const IfaceSeq seq = iface_seq(d);
    const uint32_t n = seq.e[PREV_LISTS - 1];
    // three rounds where that still gives each of the launch's warps (up to
    // four per scheduler of the GPU) something to do
    const int sub = 4u * (n / 30u) >= min(vb.nx * (blockDim.x >> 5), 4u * 608u) ? 3 : 1;
    uint32_t first, stride;
    list_span(vb, n, 10u * sub, first, stride);
    for (uint32_t w0 = first; w0 < n; w0 += stride) {
        // lane l's cell of the 30 (10): its index, whether it is (still) an
        // interface cell, its mass
        const uint32_t itl = w0 + (uint32_t)min(lane, 10 * sub - 1);
        const uint32_t il = iface_cell(d, seq, min(itl, n - 1));
        const bool vl = lane < 10 * sub && itl < n && (d.flags[il] & CL_MASK) == CL_I;
        const double m_old = d.m[il];  // requested with the populations
        float dml = 0.0f, drsl = 0.0f;
        unsigned lgl = 0;
#pragma unroll 1
        for (int turn = 0; turn < sub; ++turn) {
        const uint32_t i32 = __shfl_sync(FULL, il, 10 * turn + g);  // the float storages hold N * 19 < 2^32 elements
        const int vg = __shfl_sync(FULL, (int)vl, 10 * turn + g);  // every lane takes part
        const bool valid = lane_ok && vg != 0;
        if (!__any_sync(FULL, valid)) continue;
        const long long i = i32;
        const int x = (int)(i32 % (uint32_t)d.nx);
        const uint32_t yz = i32 / (uint32_t)d.nx;
        const int y = (int)(yz % (uint32_t)d.ny), z = (int)(yz / (uint32_t)d.ny);
        // every load of the cell in one round, independent of the neighbour
        // classes: a source beyond a wall reads the cell itself (unused), so
        // no load waits on another and none sits behind a branch
        const float phx = __ldg(d.phifsrc + i);
        float foa[3], fob[3], pa[3], pb[3], ha[3], hb[3];
        int sa[3], sb[3], ca[3], cb[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            foa[k] = trio_ld<S>(d.fsrc, TRIO_QA(k), i32, N);
            fob[k] = trio_ld<S>(d.fsrc, TRIO_QB(k), i32, N);
            sa[k] = nbr32(d, x, y, z, -TRIO_EX(k), -TRIO_EY(k), -TRIO_EZ(k));
            sb[k] = nbr32(d, x, y, z, TRIO_EX(k), TRIO_EY(k), TRIO_EZ(k));
            const uint32_t la = sa[k] < 0 ? i32 : (uint32_t)sa[k], lb = sb[k] < 0 ? i32 : (uint32_t)sb[k];
            ca[k] = __ldg(d.flags + la) & CL_MASK;
            cb[k] = __ldg(d.flags + lb) & CL_MASK;
            pa[k] = trio_ld<S>(d.fsrc, TRIO_QA(k), la, N);
            pb[k] = trio_ld<S>(d.fsrc, TRIO_QB(k), lb, N);
            ha[k] = __ldg(d.phifsrc + la);
            hb[k] = __ldg(d.phifsrc + lb);
        }
        const float fo0 = r == 0 ? P::ld(d.fsrc, 0, i, N) : 0.0f;
        // density and the velocity of the last collision (own populations)
        float drx = fo0, j0 = 0.0f, j1 = 0.0f, j2 = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            drx += foa[k] + fob[k];
            const float df = foa[k] - fob[k];
            j0 += (float)TRIO_EX(k) * df;
            j1 += (float)TRIO_EY(k) * df;
            j2 += (float)TRIO_EZ(k) * df;
        }
        drx = trio_sum(drx, b3);
        j0 = trio_sum(j0, b3);
        j1 = trio_sum(j1, b3);
        j2 = trio_sum(j2, b3);
        const float rx = 1.0f + drx;
        const float irx = __frcp_rn(rx);
        const float ux = j0 * irx - ax, uy = j1 * irx - ay, uz = j2 * irx - az;
        // the arriving populations: pull, Eq. noslip from an obstacle or a
        // wall, gas sources reconstructed below; the mass exchange of the link
        // back to a liquid or interface source; the fill level seen there
        float fpa[3], fpb[3], dm = 0.0f, fsa = phx, fsb = phx;
        unsigned solid = 0, gas = 0, seen_lg = 0;  // per direction slot 2k (a), 2k + 1 (b)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int q = s ? TRIO_QB(k) : TRIO_QA(k);
                const int si = s ? sb[k] : sa[k];
                const int ns = si < 0 ? CL_WALL : (s ? cb[k] : ca[k]);
                const float pq = s ? pb[k] : pa[k];
                const float phy = s ? hb[k] : ha[k];
                const float fbar = s ? foa[k] : fob[k];  // own population of the opposite direction
                const unsigned bit = 1u << (2 * k + s);
                const bool sol = ns == CL_WALL || ns == CL_O, gs = ns == CL_G, lq = ns == CL_L;
                // selects rather than branches: the lanes of a warp meet every
                // class, and branches would run one after another; only the
                // moving-solid term (rare) is behind a branch
                float cuw = 0.0f;
                if (ns == CL_O || (sol && d.walls_move))
                    cuw = ns == CL_O ? link_cuw_f(d, d.bodies[d.bid[si]], x, y, z, q) : (float)wall_cuw(d, x, y, z, q);
                seen_lg |= lq ? 1u : (gs ? 2u : 0u);
                solid |= sol ? bit : 0u;
                gas |= gs ? bit : 0u;
                const float fv = sol ? fbar + 6.0f * (k == 0 ? wf(1) : wf(7)) * cuw * rx : (gs ? 0.0f : pq);
                const float wgt = lq ? 1.0f : 0.5f * (phx + phy);
                dm += (sol || gs) ? 0.0f : wgt * (pq - fbar);
                const float seen = sol ? phx : (gs ? 0.0f : (lq ? 1.0f : phy));
                if (s) fpb[k] = fv;
                else fpa[k] = fv;
                if (k == 0) {
                    if (s) fsb = seen;
                    else fsa = seen;
                }
            }
        }
        // normal n = -grad(phi): component r from the member's axis pair
        // (W/E pull from x + e_x / x - e_x, N/S from x - e_y / x + e_y, T/B
        // from x - e_z / x + e_z)
        const float nvr = r == 0 ? 0.5f * (fsb - fsa) : 0.5f * (fsa - fsb);
        const float nv0 = __shfl_sync(FULL, nvr, b3), nv1 = __shfl_sync(FULL, nvr, b3 + 1),
                    nv2 = __shfl_sync(FULL, nvr, b3 + 2);
        float drg = d.drg_f;
        if (d.sigma != 0.0) {
            // gas density raised by the Laplace pressure
            const float len = sqrtf((nv0 * nv0 + nv1 * nv1) + nv2 * nv2);
            const float nur = len > 0.0f ? (r == 0 ? nv0 : (r == 1 ? nv1 : nv2)) / len : 0.0f;
            const float kap = 0.25f * trio_sum(curvature_axis_f(d, x, y, z, r, nur), b3);
            drg = d.drg_f + (6.0f * d.sigma_f) * kap;
        }
        // Eq. reconstruct for gas-sourced directions and every non-solid
        // direction with c.n below the dead band
        const float usq = ux * ux + uy * uy + uz * uz;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float cn = (float)TRIO_EX(k) * nv0 + (float)TRIO_EY(k) * nv1 + (float)TRIO_EZ(k) * nv2;  // c_a . n
            const float cu = (float)TRIO_EX(k) * ux + (float)TRIO_EY(k) * uy + (float)TRIO_EZ(k) * uz;
            const float w = k == 0 ? wf(1) : wf(7);
            const float fe = feq_dev_cu(w, cu, usq, drg) + feq_dev_cu(w, -cu, usq, drg);
            const unsigned ba = 1u << (2 * k), bb = 2u << (2 * k);
            if ((gas & ba) || (cn < -d.deadband_f && !(solid & ba))) fpa[k] = fe - fob[k];
            if ((gas & bb) || (-cn < -d.deadband_f && !(solid & bb))) fpb[k] = fe - foa[k];
        }
        dm = trio_sum(dm, b3);
        // BGK + Luo force on the deviations (the pair split of collide_store_v)
        const float fp0 = r == 0 ? fo0 : 0.0f;
        float dr = fp0, k0 = 0.0f, k1 = 0.0f, k2 = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dr += fpa[k] + fpb[k];
            const float df = fpa[k] - fpb[k];
            k0 += (float)TRIO_EX(k) * df;
            k1 += (float)TRIO_EY(k) * df;
            k2 += (float)TRIO_EZ(k) * df;
        }
        dr = trio_sum(dr, b3);
        k0 = trio_sum(k0, b3);
        k1 = trio_sum(k1, b3);
        k2 = trio_sum(k2, b3);
        const float rho = 1.0f + dr;
        const float inv = __frcp_rn(rho);
        const float vx = k0 * inv, vy = k1 * inv, vz = k2 * inv;
        const float nusq15 = (vx * vx + vy * vy + vz * vz) * -1.5f;
        const float nua3 = (vx * ax + vy * ay + vz * az) * -3.0f;
        const float om = d.omega_f, om1 = 1.0f - om;
        void *gdst = d.fdst;
        float rest = 0.0f, drs = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float w = k == 0 ? wf(1) : wf(7);
            const float wdr = dr * w, wr = rho * w, wr3 = wr * 3.0f;
            // p = the member with the positive leading component, m the other
            const float sgk = TRIO_POS(k) ? 1.0f : -1.0f;
            const float cpx = sgk * (float)TRIO_EX(k), cpy = sgk * (float)TRIO_EY(k), cpz = sgk * (float)TRIO_EZ(k);
            const float cu = cpx * vx + cpy * vy + cpz * vz;
            const float ca = cpx * ax + cpy * ay + cpz * az;
            const float A = fmaf(wr, fmaf(cu * cu, 4.5f, nusq15), wdr);
            const float C = wr * fmaf(cu, 9.0f * ca, nua3);
            const float E = fmaf(A, om, C);
            const float G = fmaf(wr3 * cu, om, wr3 * ca);
            const bool a_is_p = TRIO_POS(k) != 0;
            const float fp_p = a_is_p ? fpa[k] : fpb[k], fp_m = a_is_p ? fpb[k] : fpa[k];
            const float dnp = fmaf(fp_p, om1, E + G), dnm = fmaf(fp_m, om1, E - G);
            const int qp = a_is_p ? TRIO_QA(k) : TRIO_QB(k), qm = a_is_p ? TRIO_QB(k) : TRIO_QA(k);
            float stp = dnp, stm = dnm;
            if (valid) {
                stp = trio_st<S>(gdst, qp, i32, N, dnp);
                stm = trio_st<S>(gdst, qm, i32, N, dnm);
            }
            rest += (fp_p - stp) + (fp_m - stm);
            drs += stp + stm;
        }
        rest = trio_sum(rest, b3);
        if (r == 0) {
            const float st0 = fp0 + rest;
            if (valid) P::st_one(gdst, 0, i, N, st0);
            drs += st0;
        }
        drs = trio_sum(drs, b3);
        const unsigned lg = __shfl_sync(FULL, seen_lg, b3) | __shfl_sync(FULL, seen_lg, b3 + 1) |
                            __shfl_sync(FULL, seen_lg, b3 + 2);
        if (valid && r == 0 && (!(rho > 0.0f) || !(rho < 1e30f))) atomicOr(d.status, ST_NONFINITE);
        // to the lane that does the cell's mass update
        const int from = 3 * min(max(lane - 10 * turn, 0), 9);
        const float dmx = __shfl_sync(FULL, dm, from), drx2 = __shfl_sync(FULL, drs, from);
        const unsigned lgx = __shfl_sync(FULL, lg, from);
        if (lane >= 10 * turn && lane < 10 * turn + 10) {
            dml = dmx;
            drsl = drx2;
            lgl = lgx;
        }
        }
        const bool has_l = lgl & 1u, has_g = lgl & 2u;
        uint8_t mk = 0;
        if (vl) {
            const double m_new = m_old + (double)dml;
            const double phin = m_new / (1.0 + (double)drsl);
            d.m[il] = m_new;
            d.phidst[il] = phin;
            d.phifdst[il] = (float)phin;
            mk = phin >= 1.0 + d.eps ? MK_FILLED : (phin <= -d.eps ? MK_EMPTIED : 0);
            // an interface cell without a liquid neighbour empties, one without
            // a gas neighbour fills
            if (!mk && d.nb_rule) mk = (!has_l && has_g) ? MK_EMPTIED : ((!has_g && has_l) ? MK_FILLED : 0);
            if (mk) d.cmark[il] = mk;
        }
        const uint32_t i32 = il;
        wl_append(d, mk == MK_FILLED, WL_FILLED, i32);
        wl_append(d, mk == MK_EMPTIED, WL_EMPTIED, i32);
    }
}
#undef TRIO_QA
#undef TRIO_QB
#undef TRIO_EX
#undef TRIO_EY
#undef TRIO_EZ
#undef TRIO_POS

// ---- C1 + C2 for interface cells (Sec. 2.2): reconstruction, mass exchange.
// Double storage: one thread per cell, every sum in the order of the oracle.
__device__ __forceinline__ void interface_d(const Dev &d, const VB &vb) {
    using P = Sto<0>;
    const long long N = d.N;
    const IfaceSeq seq = iface_seq(d);
    const uint32_t n = seq.e[PREV_LISTS - 1];
    uint32_t first, stride;
    list_span(vb, n, 32u, first, stride);
    for (uint32_t it = first + (threadIdx.x & 31u); it < n; it += stride) {
        const long long i = iface_cell(d, seq, it);
        if (clsv(d, i) != CL_I) continue;
        int x, y, z;
        coords(d, i, x, y, z);
        double own_phi = d.phisrc[i];
        long long src[Q];
        int scl[Q];
        bool has_l = false, has_g = false;  // any liquid / gas among the 18 neighbours
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            src[q] = nbr(d, x, y, z, -cx(q), -cy(q), -cz(q));
            scl[q] = cls(d, src[q]);
            has_l = has_l || scl[q] == CL_L;
            has_g = has_g || scl[q] == CL_G;
        }
        // normal n = -grad(phi), central differences
        double nv[3];
        {
            double pm = fill_seen(d, nbr(d, x, y, z, -1, 0, 0), own_phi);
            double pp = fill_seen(d, nbr(d, x, y, z, 1, 0, 0), own_phi);
            nv[0] = 0.5 * (pm - pp);
            pm = fill_seen(d, nbr(d, x, y, z, 0, -1, 0), own_phi);
            pp = fill_seen(d, nbr(d, x, y, z, 0, 1, 0), own_phi);
            nv[1] = 0.5 * (pm - pp);
            pm = fill_seen(d, nbr(d, x, y, z, 0, 0, -1), own_phi);
            pp = fill_seen(d, nbr(d, x, y, z, 0, 0, 1), own_phi);
            nv[2] = 0.5 * (pm - pp);
        }
        double fo[Q], fp[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) fo[q] = P::ld(d.fsrc, q, i, N);
        double rho_x = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) rho_x += fo[q];
        double j0 = 0.0, j1 = 0.0, j2 = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (cx(q)) j0 += cx(q) * fo[q];
            if (cy(q)) j1 += cy(q) * fo[q];
            if (cz(q)) j2 += cz(q) * fo[q];
        }
        double ux[3] = {j0 / rho_x - d.a[0], j1 / rho_x - d.a[1], j2 / rho_x - d.a[2]};
        // gas density of the boundary condition, raised by the Laplace pressure
        double rg = d.rho_g;
        if (d.sigma != 0.0) {
            double nc[3];
            unit_vec_d(nv, nc);
            rg = d.rho_g + (6.0 * d.sigma) * curvature_d(d, x, y, z, nc[0], nc[1], nc[2]);
        }
        // the equilibrium sum f_eq,q + f_eq,qbar of the reconstruction is the
        // same for both members of a pair: once per pair, with the
        // collision's shared terms (collide_d_t), instead of up to four
        // evaluations per direction
        const double us15 = 1.5 * ((ux[0] * ux[0] + ux[1] * ux[1]) + ux[2] * ux[2]);
        const double wg1 = wd(1) * rg, wg2 = wd(7) * rg;
        double pull[Q], feb[Q];
#pragma unroll
        for (int q = 1; q < Q; ++q) pull[q] = (scl[q] == CL_L || scl[q] == CL_I) ? P::ld(d.fsrc, q, src[q], N) : 0.0;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            if (opp(q) < q) continue;
            double cu = 0.0, cn = 0.0;
            bool first = true;
            if (cx(q)) {
                cu = cx(q) > 0 ? ux[0] : -ux[0];
                cn = cx(q) > 0 ? nv[0] : -nv[0];
                first = false;
            }
            if (cy(q)) {
                cu = first ? (cy(q) > 0 ? ux[1] : -ux[1]) : (cy(q) > 0 ? cu + ux[1] : cu - ux[1]);
                cn = first ? (cy(q) > 0 ? nv[1] : -nv[1]) : (cy(q) > 0 ? cn + nv[1] : cn - nv[1]);
                first = false;
            }
            if (cz(q)) {
                cu = first ? (cz(q) > 0 ? ux[2] : -ux[2]) : (cz(q) > 0 ? cu + ux[2] : cu - ux[2]);
                cn = first ? (cz(q) > 0 ? nv[2] : -nv[2]) : (cz(q) > 0 ? cn + nv[2] : cn - nv[2]);
            }
            const double c3 = 3.0 * cu, s = (4.5 * cu) * cu, wg = q <= 6 ? wg1 : wg2;
            feb[q] = wg * (((1.0 + c3) + s) - us15) + wg * (((1.0 - c3) + s) - us15);
            feb[opp(q)] = cn;  // the pair's second slot carries c_q . n
        }
        fp[0] = fo[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const int qb = opp(q);
            const bool lead = qb > q;
            const double fe2 = lead ? feb[q] : feb[qb], cn = lead ? feb[qb] : -feb[q];
            if (scl[q] == CL_WALL || scl[q] == CL_O) {
                double cuw = scl[q] == CL_O ? link_cuw(d, d.bodies[d.bid[src[q]]], x, y, z, q)
                                            : (d.walls_move ? wall_cuw(d, x, y, z, q) : 0.0);
                fp[q] = fo[qb] + ((6.0 * wd(q)) * rho_x) * cuw;
            } else if (scl[q] == CL_G || cn < -d.deadband) {
                fp[q] = fe2 - fo[qb];
            } else {
                fp[q] = pull[q];
            }
        }
        // mass exchange with the neighbour x + c_q: the source of qbar, whose
        // class and population are at hand
        double dm = 0.0;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const int qb = opp(q);
            if (scl[qb] == CL_L) {
                dm += pull[qb] - fo[q];
            } else if (scl[qb] == CL_I) {
                const double wgt = 0.5 * (own_phi + d.phisrc[src[qb]]);
                dm += wgt * (pull[qb] - fo[q]);
            }
        }
        const double m_new = d.m[i] + dm;
        double fn[Q];
        collide_d(d, fp, fn);
        double r = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            P::st(d.fdst, q, i, N, fn[q]);
            r += fn[q];
        }
        double phin = m_new / r;
        d.m[i] = m_new;
        d.phidst[i] = phin;
        if (!(r == r) || r <= 0.0) atomicOr(d.status, ST_NONFINITE);
        uint8_t mk = phin >= 1.0 + d.eps ? MK_FILLED : (phin <= -d.eps ? MK_EMPTIED : 0);
        // an interface cell without a liquid neighbour empties, one without
        // a gas neighbour fills
        if (!mk && d.nb_rule) mk = (!has_l && has_g) ? MK_EMPTIED : ((!has_g && has_l) ? MK_FILLED : 0);
        if (mk) d.cmark[i] = mk;
        wl_append(d, mk == MK_FILLED, WL_FILLED, (uint32_t)i);
        wl_append(d, mk == MK_EMPTIED, WL_EMPTIED, (uint32_t)i);
    }
}
template <int S> __device__ __forceinline__ void interface_body(const Dev &d, const VB &vb) {
    if constexpr (S == 0) interface_d(d, vb);
    else interface_trio<S>(d, vb);
}
template <int S>
__global__ void __launch_bounds__(128, S == 0 ? 2 : LBMFS_IFACE_MINB) k_interface(const __grid_constant__ Dev d) {
    interface_body<S>(d, vb_own());
}

// ------------------------------------------------- C3: conversions (Sec. 2.2)

// The conversion bodies take a warp per listed cell, lane q its neighbour in
// direction q: the classes, marks and atomics of the 18 neighbours are in
// flight together (one thread per cell issued its atomics one after another),
// and the cells a warp marks are appended with one reservation.  The warps of
// a short list go to different SMs.
// (`skip` items of other lists that the same phase works on come first: the
// lists share the warps instead of all starting at the first one)
#define WARP_LOOP(L, var, skip)                                                                                \
    const uint32_t n_##var = wl_count(d, L), w_##var = vb.nx * (blockDim.x >> 5), s_##var = (skip) % w_##var;   \
    for (uint32_t it_##var = ((threadIdx.x >> 5) * vb.nx + vb.x + w_##var - s_##var) % w_##var; it_##var < n_##var; \
         it_##var += w_##var)

// set mark `bit` on the lanes' cells (want) and append those newly marked
__device__ __forceinline__ void mark_append(const Dev &d, bool want, long long yi, uint8_t bit, int list) {
    const bool nw = want && !(mark_or(d, yi, bit) & bit);
    __syncwarp();
    wl_append(d, nw, list, (uint32_t)yi);
}

// gas neighbours of filled cells become interface
__device__ __forceinline__ void conv_filled_body(const Dev &d, const VB &vb) {
    const int lane = threadIdx.x & 31;
    WARP_LOOP(WL_FILLED, a, 0u) {
        int x, y, z;
        coords(d, d.list[WL_FILLED][it_a], x, y, z);
        const long long yi = lane_nbr(d, lane, x, y, z);
        mark_append(d, cls(d, yi) == CL_G, yi, MK_NEWG, WL_NEWG);
    }
}

// an emptied cell next to a filled one is kept; liquid neighbours of the others
// become interface
__device__ __forceinline__ void conv_emptied_body(const Dev &d, const VB &vb) {
    const int lane = threadIdx.x & 31;
    WARP_LOOP(WL_EMPTIED, a, wl_count(d, WL_FILLED)) {
        const long long i = d.list[WL_EMPTIED][it_a];
        int x, y, z;
        coords(d, i, x, y, z);
        const long long yi = lane_nbr(d, lane, x, y, z);
        const int mk = yi >= 0 ? d.cmark[yi] : 0, c = cls(d, yi);
        if (__any_sync(0xffffffffu, (mk & MK_FILLED) != 0)) {
            if (lane == 0) mark_and(d, i, MK_EMPTIED);
            continue;
        }
        mark_append(d, c == CL_L, yi, MK_NEWL, WL_NEWL);
    }
}

// density of a cell by a whole warp: lane q loads population q, the sum is
// taken in q order (as cell_density takes it) on every lane
template <int S> __device__ __forceinline__ double warp_density(const Dev &d, const void *g, long long i) {
    const int lane = threadIdx.x & 31;
    typename Sto<S>::R v = 0, r = 0;
    if (lane < Q) v = Sto<S>::ld(g, lane, i, d.N);
#pragma unroll
    for (int q = 0; q < Q; ++q) r += __shfl_sync(0xffffffffu, v, q);
    if constexpr (S != 0) return 1.0 + (double)r;
    else return r;
}

// new interface cells: from gas f = f_eq(mean rho, mean u) of the liquid and
// interface neighbours, m = 0; from liquid m = rho
// f_eq of the lane's direction; the products by the components are exact, so
// this is feq_d for every q
__device__ __forceinline__ double feq_lane(int q, double rho, const double *u) {
    const double ex = (double)dir_x(q), ey = (double)dir_y(q), ez = (double)dir_z(q);
    const double cu = (ex * u[0] + ey * u[1]) + ez * u[2];
    const double usq = (u[0] * u[0] + u[1] * u[1]) + u[2] * u[2];
    const double t = ((1.0 + 3.0 * cu) + (4.5 * cu) * cu) - 1.5 * usq;
    return ((q == 0 ? wd(0) : (q <= 6 ? wd(1) : wd(7))) * rho) * t;
}
// store the cell whose population q lane q holds as f (Sto::st_cell by a warp)
template <int S> __device__ __forceinline__ void warp_store_cell(const Dev &d, long long i, int lane, double f) {
    if constexpr (S == 0) {
        if (lane < Q) Sto<0>::st(d.fdst, lane, i, d.N, f);
    } else {
        const float dv = (float)(f - (lane == 0 ? wd(0) : (lane <= 6 ? wd(1) : wd(7))));
        if constexpr (S == 1) {
            if (lane < Q) Sto<1>::st(d.fdst, lane, i, d.N, dv);
        } else {
            // the rest population takes up what the others lose in rounding
            float lost = 0.0f;
            if (lane >= 1 && lane < Q) lost = dv - Sto<2>::st_one(d.fdst, lane, i, d.N, dv);
            float rest = 0.0f;
#pragma unroll
            for (int q = 1; q < Q; ++q) rest += __shfl_sync(0xffffffffu, lost, q);
            if (lane == 0) Sto<2>::st_one(d.fdst, 0, i, d.N, dv + rest);
        }
    }
}
template <int S>
__device__ __forceinline__ void conv_init_body(const Dev &d, const VB &vb) {
    {
        // one warp per new cell: lane q reads neighbour q (all neighbours'
        // populations in flight together), the sums are taken in q order
        // from the gathered values, lane q evaluates f_eq,q
        const int lane = threadIdx.x & 31;
        WARP_LOOP(WL_NEWG, w, 0u) {
            const long long i = d.list[WL_NEWG][it_w];
            int x, y, z;
            coords(d, i, x, y, z);
            if (lane == 0 && z > *d.ztop_wr + ZTOP_MARGIN) atomicOr(d.status, ST_TOP);
            double r = 0.0, u[3] = {0.0, 0.0, 0.0};
            int fluid = 0;
            if (lane >= 1 && lane < Q) {
                const long long zi = nbr(d, x, y, z, cx(lane), cy(lane), cz(lane));
                const int zc = cls(d, zi);
                if (zc == CL_L || zc == CL_I) {
                    fluid = 1;
                    r = cell_rho_u<S>(d, d.fdst, zi, u);
                }
            }
            // lane c < 4 sums component c (density, velocity) in q order; lane q
            // evaluates f_eq,q and stores population q
            const unsigned fm = __ballot_sync(0xffffffffu, fluid != 0);
            double sum = 0.0;
            for (unsigned m = fm; m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                const double rq = __shfl_sync(0xffffffffu, r, q), u0 = __shfl_sync(0xffffffffu, u[0], q),
                             u1 = __shfl_sync(0xffffffffu, u[1], q), u2 = __shfl_sync(0xffffffffu, u[2], q);
                sum += lane == 0 ? rq : (lane == 1 ? u0 : (lane == 2 ? u1 : u2));
            }
            const double mean = sum / __popc(fm);
            const double rm = __shfl_sync(0xffffffffu, mean, 0);
            const double um[3] = {__shfl_sync(0xffffffffu, mean, 1), __shfl_sync(0xffffffffu, mean, 2),
                                  __shfl_sync(0xffffffffu, mean, 3)};
            warp_store_cell<S>(d, i, lane, feq_lane(lane, rm, um));
            if (lane == 0) d.m[i] = 0.0;
        }
    }
    {
        LIST_LOOP(WL_NEWL, b) {
            const long long i = d.list[WL_NEWL][it_b];
            d.m[i] = cell_density<S>(d, d.fdst, i);
        }
    }
}

// the new classes
__device__ __forceinline__ void conv_flags_body(const Dev &d, const VB &vb) {
    {
        LIST_LOOP(WL_FILLED, a) set_cls(d, d.list[WL_FILLED][it_a], CL_L);
    }
    {
        LIST_LOOP(WL_EMPTIED, b) {
            long long i = d.list[WL_EMPTIED][it_b];
            if (d.cmark[i] & MK_EMPTIED) set_cls(d, i, CL_G);
        }
    }
    {
        LIST_LOOP(WL_NEWG, c) set_cls(d, d.list[WL_NEWG][it_c], CL_I);
    }
    {
        LIST_LOOP(WL_NEWL, e) set_cls(d, d.list[WL_NEWL][it_e], CL_I);
    }
}

// the class a cell of class c has after the conversions, by its marks
__device__ __forceinline__ int class_after(int c, int mk) {
    return mk & (MK_NEWG | MK_NEWL) ? CL_I : (mk & MK_FILLED ? CL_L : (mk & MK_EMPTIED ? CL_G : c));
}

// interface neighbours of converted cells receive excess mass.  The
// converted cell's share e(x) / k(x) is computed here, once, and kept in its
// mass entry (a converted cell is liquid or gas now, so the entry is not read
// as a mass again before the cell next becomes interface, which sets it); the
// mass of a cell without interface neighbours goes to the lost-mass ledger
template <int S>
__device__ __forceinline__ void claim_receivers(const Dev &d, int lane, long long i, uint8_t mk) {
    int x, y, z;
    coords(d, i, x, y, z);
    const long long yi = lane_nbr(d, lane, x, y, z);
    // (the classes themselves change in the next phase, beside the excess)
    const bool want = yi >= 0 && class_after(clsv(d, yi), d.cmark[yi]) == CL_I;
    const double m = d.m[i];
    const int k = __popc(__ballot_sync(0xffffffffu, want));
    const double e = (mk & MK_FILLED) ? m - warp_density<S>(d, d.fdst, i) : m;
    if (lane == 0) {
        if (k > 0) d.m[i] = e / k;
        else atomicAdd(&d.ledger[LG_LOST], e);
    }
    __syncwarp();
    mark_append(d, want, yi, MK_RECV, WL_RECV);
}

template <int S>
__device__ __forceinline__ void conv_claim_body(const Dev &d, const VB &vb) {
    const int lane = threadIdx.x & 31;
    {
        WARP_LOOP(WL_FILLED, a, wl_count(d, WL_NEWG)) claim_receivers<S>(d, lane, d.list[WL_FILLED][it_a], MK_FILLED);
    }
    {
        WARP_LOOP(WL_EMPTIED, b, wl_count(d, WL_NEWG) + wl_count(d, WL_FILLED)) {
            const long long i = d.list[WL_EMPTIED][it_b];
            const uint8_t mk = d.cmark[i];
            if (mk & MK_EMPTIED) claim_receivers<S>(d, lane, i, mk);
        }
    }
}

// Receivers gather e(x) / k(x) over their converted neighbours in q order: the
// neighbours' marks, then the converted ones' shares (computed when the
// receivers were claimed).  A warp per receiver with a lane per neighbour while
// there are warps for it (a thread's thousand instructions for its 18
// neighbours, at the rate of a lone warp, took 10 us for a single receiver); a
// thread each for the long lists of large tanks.
template <int S> __device__ __forceinline__ void set_mass(const Dev &d, long long i, double m, double rho) {
    d.m[i] = m;
    const double ph = m / rho;
    d.phidst[i] = ph;
    if constexpr (S != 0) d.phifdst[i] = (float)ph;
}
template <int S>
__device__ __forceinline__ void conv_excess_body(const Dev &d, const VB &vb) {
    if (wl_count(d, WL_RECV) <= 2u * vb.nx * (blockDim.x >> 5)) {
        const int lane = threadIdx.x & 31;
        WARP_LOOP(WL_RECV, w, 0u) {
            const long long i = d.list[WL_RECV][it_w];
            int x, y, z;
            coords(d, i, x, y, z);
            const long long yi = lane_nbr(d, lane, x, y, z);
            const bool conv = yi >= 0 && (d.cmark[yi] & (MK_FILLED | MK_EMPTIED));
            const double share = conv ? d.m[yi] : 0.0, m = d.m[i], rho = warp_density<S>(d, d.fdst, i);
            double acc = 0.0;
            for (unsigned b = __ballot_sync(0xffffffffu, conv); b; b &= b - 1)
                acc += __shfl_sync(0xffffffffu, share, __ffs(b) - 1);
            if (lane == 0) set_mass<S>(d, i, m + acc, rho);
            __syncwarp();
        }
        return;
    }
    LIST_LOOP(WL_RECV, a) {
        long long i = d.list[WL_RECV][it_a];
        int x, y, z;
        coords(d, i, x, y, z);
        unsigned cm = 0;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            long long yi = nbr(d, x, y, z, cx(q), cy(q), cz(q));
            if (yi >= 0 && (d.cmark[yi] & (MK_FILLED | MK_EMPTIED))) cm |= 1u << q;
        }
        const double rho = cell_density<S>(d, d.fdst, i);
        double acc = 0.0;
        for (unsigned b = cm; b; b &= b - 1) {
            const int q = __ffs(b) - 1;
            acc += d.m[nbr(d, x, y, z, dir_x(q), dir_y(q), dir_z(q))];
        }
        set_mass<S>(d, i, d.m[i] + acc, rho);
    }
}

// marks are cleared; bit by bit where the remap may be marking covered cells at
// the same time (shared; the atomics take 0.8 us longer)
__device__ __forceinline__ void conv_finish_body(const Dev &d, const VB &vb, bool shared) {
    const int lists[5] = {WL_FILLED, WL_EMPTIED, WL_NEWG, WL_NEWL, WL_RECV};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        LIST_LOOP(lists[k], a) {
            const long long i = d.list[lists[k]][it_a];
            if (shared) mark_and(d, i, MK_FILLED | MK_EMPTIED | MK_NEWG | MK_NEWL | MK_RECV);
            else d.cmark[i] = 0;
        }
    }
}

// ----------------------------------------------- C5: rigid-body update
// (the role the paper gives the pe engine, Sec. 2.3: the body moves under the
// hydrodynamic force and torque and gravity; the paper does not give the
// integrator, this one is a virtual-mass explicit update)

// One warp per body: the fixed-order sum of the force partials, then the
// update.  A double operation holds the scheduler for 64 cycles and a division
// for 550 whatever the number of active lanes, so the update is written for
// lanes: lane l works on component k = l % 3 of the vectors, lanes with
// (l / 3) odd on the rotation where it mirrors the translation, and lanes 0..8
// on the nine entries of a rotation matrix.  Every value is the scalar update's
// (one thread, about 700 double operations, 22 us; now about 80 and four
// divisions), rounded the same way: this unit is compiled without fused
// multiply-add.
__device__ __forceinline__ double lane_of(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
// (a_0 + a_1) + a_2 of the values that lanes base .. base + 2 hold
__device__ __forceinline__ double sum3(double a, int base) {
    return (lane_of(a, base) + lane_of(a, base + 1)) + lane_of(a, base + 2);
}
// entry lane (row-major, lanes 0..8) of the rotation matrix of the quaternion
// whose component j lane j holds (see rotation)
__device__ __forceinline__ double rotation_lane(double q, int lane) {
    const int e = lane < 9 ? lane : 0, i = e / 3, j = e - 3 * i;
    const bool diag = i == j;
    // diagonal: 1 - 2 (a a + b b) with the two other axes; else 2 (x_i x_j +- w x_k)
    const int o1 = i == 0 ? 1 : 0, o2 = i == 2 ? 1 : 2, k = 3 - i - j;
    const bool neg = !diag && (j - i + 3) % 3 == 1;
    const double p1 = lane_of(q, 1 + (diag ? o1 : i)) * lane_of(q, 1 + (diag ? o1 : j));
    const double p2 = lane_of(q, diag ? 1 + o2 : 0) * lane_of(q, 1 + (diag ? o2 : k));
    const double r = 2.0 * (p1 + (neg ? -p2 : p2));
    return diag ? 1.0 - r : r;
}
__device__ __forceinline__ void bodies_body(const Dev &d, const VB &vb) {
    const int bi = vb.x, lane = threadIdx.x & 31;
    const Body &b = d.bodies[bi];
    Body &nb = d.bodies_new[bi];
    static_assert(sizeof(Body) % 8 == 0, "body records are copied in 8-byte words");
    for (int w = lane; w < (int)(sizeof(Body) / 8); w += 32)
        reinterpret_cast<unsigned long long *>(&nb)[w] = reinterpret_cast<const unsigned long long *>(&b)[w];
    double tot;  // lane c < 7 holds sum c: force, torque, |terms|
    const int k = lane % 3, k1 = k == 2 ? 0 : k + 1, k2 = k == 0 ? 2 : k - 1;
    const bool rot = (lane / 3) & 1;
    if (d.part128) {
        // double storage: exact 128-bit partials (fixed96), summed exactly
        const unsigned long long *pp = reinterpret_cast<const unsigned long long *>(d.part);
        unsigned __int128 mine = 0;
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            unsigned __int128 v = 0;
            for (int j = lane; j < FORCE_BLOCKS; j += 32) {
                const long long at = 2 * (((long long)bi * FORCE_BLOCKS + j) * 7 + c);
                v += ((unsigned __int128)pp[at + 1] << 64) | (unsigned __int128)pp[at];
            }
            for (int off = 16; off > 0; off >>= 1) v += shfl_xor_128(v, off);
            if ((lane & 7) == c) mine = v;
        }
        tot = fixed96_value(mine);
    } else {
        static_assert(FORCE_BLOCKS == 64, "two partials per lane");
        // tree sums (lane l + lane l + off) of the seven components packed so
        // that each level halves the registers: 9 additions instead of 35
        double v[8];
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            const double *p = d.part + ((long long)bi * FORCE_BLOCKS + lane) * 7 + c;
            v[c] = p[0] + p[32 * 7];
        }
        v[7] = 0.0;
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            const int off = 16 >> h;
            const bool up = lane & off;
#pragma unroll
            for (int c = 0; c < (8 >> h); c += 2) {
                const double send = up ? v[c] : v[c + 1], keep = up ? v[c + 1] : v[c];
                v[c / 2] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        }
        double t = v[0];
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        // component c sits where bit 4, 3, 2 of the lane are bit 0, 1, 2 of c
        const int c = lane & 7;
        tot = lane_of(t, ((c & 1) << 4) | ((c & 2) << 2) | (c & 4));
    }
    // (either way lane c holds sum c)
    const double ft = lane_of(tot, rot ? 3 + k : k), fabs_sum = lane_of(tot, 6);
    __syncwarp();
    if (lane < 3) {
        nb.F[k] = ft;
        nb.plo[k] = b.lo[k];
        nb.phi[k] = b.hi[k];
    }
    if (lane >= 3 && lane < 6) nb.T[k] = ft;
    if (lane == 0) nb.S = fabs_sum;
    const int base = b.mode & 0xff;
    if (base == 0) {
        if (lane < 3) nb.v[k] = nb.w[k] = nb.dv[k] = nb.dw[k] = 0.0;
        return;
    }
    // the update is driven by the mean of this step's and the previous step's
    // force and torque (the force alone on the first step; the force alone
    // throughout when the two-step mean is switched off): near tau = 1/2 a
    // force that flips sign every step would feed the barely damped BGK modes
    // of that period through the wall velocity
    const double ftp = rot ? b.Tp[k] : b.Fp[k];
    const double fh = d.force_mean && b.nF ? 0.5 * (ft + ftp) : ft;  // force, or torque (rot)
    const double hk = b.h[k], h0 = b.h[0], dens = b.dens, C = d.vmass;
    const double vol = b.vol, mass = b.mass, I = b.I[k];  // (set with the body)
    double q = b.q[lane & 3];
    const double R = rotation_lane(q, lane);
    const double c0 = lane_of(R, k), c1 = lane_of(R, 3 + k), c2 = lane_of(R, 6 + k);  // column k
    const double T0 = lane_of(fh, 3), T1 = lane_of(fh, 4), T2 = lane_of(fh, 5);
    const double w0 = b.w[0], w1 = b.w[1], w2 = b.w[2];
    // translation (virtual mass: Schwarz, Kempe and Froehlich 2015) and rotation
    // have the form (A + C (B D)) / (E + C B), D the last acceleration
    double A = fh + mass * d.grav[k], B = vol, E = mass, wb;
    const double Dl = rot ? (base == 2 ? b.dw[0] : b.dw[k]) : b.dv[k];
    if (base == 2) {
        // the dot products with the axis: of column k (lanes 0..2: the axis in the
        // body's frame), of the torque (lane 3) and of the angular velocity (lane 4)
        const double v0 = lane < 3 ? c0 : (lane == 3 ? T0 : w0), v1 = lane < 3 ? c1 : (lane == 3 ? T1 : w1),
                     v2 = lane < 3 ? c2 : (lane == 3 ? T2 : w2);
        const double dot = (v0 * b.axis[0] + v1 * b.axis[1]) + v2 * b.axis[2];
        const double Ia = sum3((dot * dot) * I, 0);
        const double Ifa = Ia / dens;
        wb = lane_of(dot, 4);
        const double ta = lane_of(dot, 3);
        if (rot) {
            A = ta;
            B = Ifa;
            E = Ia;
        }
    } else {
        // column k times the angular velocity (lanes 0..2) and the torque (3..5)
        const double dot = (c0 * (rot ? T0 : w0) + c1 * (rot ? T1 : w1)) + c2 * (rot ? T2 : w2);
        const double If = I / dens;
        wb = lane_of(dot, k);
        const double tb = lane_of(dot, 3 + k);
        const double L = I * wb;
        const double gy = lane_of(wb, k1) * lane_of(L, k2) - lane_of(wb, k2) * lane_of(L, k1);
        const double Ar = tb - gy;
        if (rot) {
            A = Ar;
            B = If;
            E = I;
        }
    }
    const double acc = (A + C * (B * Dl)) / (E + C * B);  // dv (lanes 0..2), dw (lanes 3..5)
    const double dv = lane_of(acc, k), dw = lane_of(acc, 3 + k);
    double v = b.v[k] + dv;
    if (b.mode & 0x100) v = v * (1.0 - b.damp);
    double w;
    if (base == 2) {
        w = (wb + lane_of(dw, 0)) * b.axis[k];
    } else {
        wb = wb + dw;
        w = (lane_of(R, 3 * k) * lane_of(wb, 0) + lane_of(R, 3 * k + 1) * lane_of(wb, 1)) +
            lane_of(R, 3 * k + 2) * lane_of(wb, 2);
    }
    const int nk = k == 0 ? d.nx : (k == 1 ? d.ny : d.nz);
    const double nn = (double)nk;
    double o = b.o[k] + v;
    if (d.periodic & (1u << k)) {
        if (o >= nn) o = o - nn;
        else if (o < 0.0) o = o + nn;
    }
    {
        // lane j < 4: component j of the quaternion's rate of change,
        //   -((w0 qx + w1 qy) + w2 qz), qw w0 + (w1 qz - w2 qy), ...
        const int j = lane & 3;
        const double v0 = lane_of(w, 0), v1 = lane_of(w, 1), v2 = lane_of(w, 2);
        const double qw = lane_of(q, 0), qx = lane_of(q, 1), qy = lane_of(q, 2), qz = lane_of(q, 3);
        const double m1 = (j == 0 ? v0 : qw) * (j == 0 ? qx : (j == 1 ? v0 : (j == 2 ? v1 : v2)));
        const double m2 = (j == 0 ? v1 : (j == 1 ? v1 : (j == 2 ? v2 : v0))) * (j == 0 ? qy : (j == 1 ? qz : (j == 2 ? qx : qy)));
        const double m3 = (j == 0 ? v2 : (j == 1 ? v2 : (j == 2 ? v0 : v1))) * (j == 0 ? qz : (j == 1 ? qy : (j == 2 ? qz : qx)));
        const double s = (j == 0 ? m1 : m2) + (j == 0 ? m2 : -m3);
        const double t = s + (j == 0 ? m3 : m1);
        const double nq = q + 0.5 * (j == 0 ? -t : t);
        const double sq = nq * nq;
        const double norm = sqrt(((lane_of(sq, 0) + lane_of(sq, 1)) + lane_of(sq, 2)) + lane_of(sq, 3));
        q = nq / norm;
    }
    // the new pose's rotation, its float copies and the cells it may cover
    const double Rn = rotation_lane(q, lane);
    const double fl = floor(o);
    const double e = b.shape == 1 ? h0
                                  : (fabs(lane_of(Rn, 3 * k)) * h0 + fabs(lane_of(Rn, 3 * k + 1)) * b.h[1]) +
                                        fabs(lane_of(Rn, 3 * k + 2)) * b.h[2];
    const double olo = o - e, ohi = o + e;
    int lo = (int)floor(olo) - 1, hi = (int)floor(ohi) + 2;
    if (!(d.periodic & (1u << k))) {
        lo = lo < 0 ? 0 : lo;
        hi = hi > nk ? nk : hi;
    } else if (hi - lo > nk) {
        hi = lo + nk;
    }
    if (hi < lo) hi = lo;
    if (lane < 9) {
        nb.R[lane] = Rn;
        nb.Rf[lane] = (float)Rn;
    }
    if (lane < 4) nb.q[lane] = q;
    if (lane == 0) nb.nF = 1;
    if (lane < 3) {
        nb.Fp[k] = ft;
        nb.dv[k] = dv;
        nb.v[k] = v;
        nb.o[k] = o;
        nb.oi[k] = (int)fl;
        nb.of[k] = (float)(o - fl);
        nb.hf[k] = (float)(b.shape == 1 && k == 0 ? h0 * h0 : hk);
        nb.lo[k] = lo;
        nb.hi[k] = hi;
        // a moving box that reaches a wall plane would need a contact model
        // (the paper's rigid-body engine); report it instead of running on
        if (!(d.periodic & (1u << k)) && (olo < 0.0 || ohi > nn)) atomicOr(d.status, ST_CONTACT);
    }
    if (lane >= 3 && lane < 6) {
        nb.Tp[k] = ft;
        if (base != 2 || k == 0) nb.dw[k] = dw;
        nb.w[k] = w;
    }
}
__global__ void k_bodies(const __grid_constant__ Dev d) {
    launch_dependents();  // the remap's scan, which waits for this launch's end
    bodies_body(d, vb_own());
}

// ----------------------------------------------- C6: remap (Sec. 2.3, 2.4)

// whether a cell lies in the body's range at its previous pose
__device__ __forceinline__ bool in_prev_range(const Dev &d, const Body &b, int x, int y, int z) {
    const int c[3] = {x, y, z}, n3[3] = {d.nx, d.ny, d.nz};
    bool in = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int t = c[k] - b.plo[k];
        if (d.periodic & (1u << k)) t = ((t % n3[k]) + n3[k]) % n3[k];
        in = in && t >= 0 && t < b.phi[k] - b.plo[k];
    }
    return in;
}
// Which cells body vb.y covers and which it leaves with its new pose: the
// obstacle set is not touched by the conversions, so the lists are made from
// it and the two poses alone, beside the bulk kernel; remap_apply_body acts on
// them once the conversions are done.  (Two scans behind the
// conversions before, 6 to 8 us each on a small tank; now one of 6 to 10 us.)
__device__ __forceinline__ void remap_scan_body(const Dev &d, const VB &vb) {
    const int bi = vb.y;
    const Body &b = d.bodies_new[bi];
    const uint32_t lane = threadIdx.x & 31u;
    // one pass over the cells of both poses' ranges (they differ by a cell or
    // two; across a periodic seam the old one is shifted to the new)
    const int n3[3] = {d.nx, d.ny, d.nz};
    int lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int shift = 0;
        if (d.periodic & (1u << k)) shift = b.plo[k] - b.lo[k] > n3[k] / 2 ? -n3[k] : (b.lo[k] - b.plo[k] > n3[k] / 2 ? n3[k] : 0);
        // (an empty range, of a body that has left the grid, adds nothing)
        const bool now = b.hi[k] > b.lo[k], was = b.phi[k] > b.plo[k];
        lo[k] = now && was ? min(b.lo[k], b.plo[k] + shift) : (now ? b.lo[k] : b.plo[k]);
        hi[k] = now && was ? max(b.hi[k], b.phi[k] + shift) : (now ? b.hi[k] : b.phi[k]);
        if ((d.periodic & (1u << k)) && hi[k] - lo[k] > n3[k]) hi[k] = lo[k] + n3[k];
        if (hi[k] < lo[k]) hi[k] = lo[k];
    }
    const uint32_t n = (uint32_t)range_count(lo, hi);
    uint32_t first, stride;
    list_span(vb, n, 32u, first, stride);
    for (uint32_t k0 = first; k0 < n; k0 += stride) {
        const uint32_t kk = k0 + lane;
        long long i = 0;
        bool cover = false, pend = false;
        if (kk < n) {
            int x, y, z;
            range_cell(d, lo, hi, kk, x, y, z);
            i = x + (long long)d.nx * (y + (long long)d.ny * z);
            const bool solid = clsv(d, i) == CL_O, own = solid && d.bid[i] == bi;
            if (!solid || own) {
                const bool in = inside(d, b, x, y, z);
                cover = !solid && in;
                pend = own && !in && (!d.loose || in_prev_range(d, b, x, y, z));
            }
        }
        if (__any_sync(0xffffffffu, cover)) wl_append(d, cover, WL_COVER, (uint32_t)i);
        // the covering body (until remap_apply_body makes the cell an obstacle
        // nothing reads its id)
        if (cover) d.bid[i] = (uint8_t)bi;
        if (__any_sync(0xffffffffu, pend)) wl_append(d, pend, WL_PEND, (uint32_t)i);
    }
}
constexpr int SCAN_THREADS = 64;
__global__ void __launch_bounds__(SCAN_THREADS) k_remap_scan(const __grid_constant__ Dev d) {
    wait_for_launch();
    remap_scan_body(d, vb_own());
}

// listed cells inside a body's new pose become obstacle, their mass is booked;
// listed obstacle cells outside it are pending.  A cell that several bodies
// cover in one step is listed once for each: it is booked once, and the first of
// those bodies has it.  (Looking for lower bodies at each covered cell in the
// scan instead: 200 spheres 257 -> 319 us per step.)
template <int S>
__device__ __forceinline__ void remap_apply_body(const Dev &d, const VB &vb) {
    {
        LIST_LOOP(WL_COVER, a) {
            const long long i = d.list[WL_COVER][it_a];
            if (d.nb > 1 && (mark_or(d, i, MK_COVER) & MK_COVER)) {
                int x, y, z, j = 0;
                coords(d, i, x, y, z);
#pragma unroll 1
                while (j < d.nb - 1 && !inside(d, d.bodies_new[j], x, y, z)) ++j;
                d.bid[i] = (uint8_t)j;
                continue;
            }
            const int c = clsv(d, i);
            const double mass = c == CL_L ? cell_density<S>(d, d.fdst, i) : (c == CL_I ? d.m[i] : 0.0);
            if (mass != 0.0) atomicAdd(&d.ledger[LG_COVERED], mass);
            set_cls(d, i, CL_O);
        }
    }
    {
        LIST_LOOP(WL_PEND, b) mark_or(d, d.list[WL_PEND][it_b], MK_PEND);
    }
}

// What a pending cell becomes (Sec. 2.4), from its numbers of liquid, interface
// and gas neighbours and their sums of density and fill level.
__device__ __forceinline__ void resolve_decide(const Dev &d, uint32_t it, int nL, int nI, int nG, double sr, double sp) {
    uint8_t dec = 0;
    if (nL > 0 && nG > 0) {
        dec = CL_I;
        d.rrho[it] = sr / (nL + nI);
        d.rphi[it] = nI > 0 ? sp / nI : 0.5;
    } else if (nG == 0 && nL + nI > 0) {
        dec = CL_L;
        d.rrho[it] = sr / (nL + nI);
    } else if (nL == 0 && nG > 0) {
        dec = CL_G;
    }
    d.rdec[it] = dec;
}
// The two halves of a pass for a long list, a thread per pending cell: the
// decision, and the cells that have one (false: undecided yet).
template <int S> __device__ __forceinline__ void resolve_look(const Dev &d, uint32_t it) {
    const long long i = d.list[WL_PEND][it];
    if (!(d.cmark[i] & MK_PEND)) {
        d.rdec[it] = 0;
        return;
    }
    int x, y, z;
    coords(d, i, x, y, z);
    // marks and classes, then the neighbours in q order
    unsigned mL = 0, mI = 0, mG = 0;
#pragma unroll 6
    for (int q = 1; q < Q; ++q) {
        const long long yi = nbr(d, x, y, z, dir_x(q), dir_y(q), dir_z(q));
        const int c = yi < 0 || (d.cmark[yi] & MK_PEND) ? 0 : clsv(d, yi);
        mL |= (c == CL_L ? 1u : 0u) << q;
        mI |= (c == CL_I ? 1u : 0u) << q;
        mG |= (c == CL_G ? 1u : 0u) << q;
    }
    double sr = 0.0, sp = 0.0;
    for (unsigned m = mL | mI; m; m &= m - 1) {
        const int q = __ffs(m) - 1;
        const long long yi = nbr(d, x, y, z, dir_x(q), dir_y(q), dir_z(q));
        sr += cell_density<S>(d, d.fdst, yi);
        if (mI & (1u << q)) sp += d.phidst[yi];
    }
    resolve_decide(d, it, __popc(mL), __popc(mI), __popc(mG), sr, sp);
}
template <int S> __device__ __forceinline__ bool resolve_set(const Dev &d, uint32_t it, bool last) {
    const long long i = d.list[WL_PEND][it];
    if (!(d.cmark[i] & MK_PEND)) return true;
    int dec = d.rdec[it];
    if (dec == 0 && last) dec = CL_G;
    if (dec == 0) return false;
    d.cmark[i] = MK_FRESH;
    set_cls(d, i, dec);
    if (dec == CL_G) return true;
    int x, y, z;
    coords(d, i, x, y, z);
    if (z > *d.ztop_wr + ZTOP_MARGIN) atomicOr(d.status, ST_TOP);
    double p[3] = {x + 0.5, y + 0.5, z + 0.5}, uw[3];
    body_velocity_at(d, d.bodies_new[d.bid[i]], p, uw);
    const double rho = d.rrho[it];
    float dv0 = 0.0f, rest = 0.0f;  // (as warp_store_cell rounds them)
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
        const double f = feq_lane(q, rho, uw);
        if constexpr (S == 0) {
            Sto<0>::st(d.fdst, q, i, d.N, f);
        } else {
            const float dv = (float)(f - (q == 0 ? wd(0) : (q <= 6 ? wd(1) : wd(7))));
            if constexpr (S == 1) Sto<1>::st(d.fdst, q, i, d.N, dv);
            else if (q == 0) dv0 = dv;
            else rest += dv - Sto<2>::st_one(d.fdst, q, i, d.N, dv);
        }
    }
    if constexpr (S == 2) Sto<2>::st_one(d.fdst, 0, i, d.N, dv0 + rest);
    const double dens = cell_density<S>(d, d.fdst, i);
    if (dec == CL_I) set_mass<S>(d, i, d.rphi[it] * rho, dens);
    d.rrho[it] = dens;  // as stored, for what follows
    return true;
}

// Jacobi passes of the obstacle-to-fluid rule over the pending cells, closure,
// uncovered-mass ledger (one block).  Up to RESOLVE_WARP pending cells a warp
// each, whose latency is short; more by a thread each: a warp's double
// operations hold their scheduler as long for one cell as for 32.  Measured, us
// of the tail with 36, 72, 150, 366 and 1145 pending cells: a warp each 75, 98,
// 169, 350 and 1032, a thread each 69, 77, 94, 127 and 307.
#ifndef LBMFS_RESOLVE_WARP
#define LBMFS_RESOLVE_WARP 36
#endif
constexpr uint32_t RESOLVE_WARP = LBMFS_RESOLVE_WARP;
template <int S>
__device__ __forceinline__ void remap_resolve_body(const Dev &d, const VB &vb) {
    uint32_t n = wl_count(d, WL_PEND);
    if (n == 0) return;
    __shared__ int s_any;
    const bool wide = n > RESOLVE_WARP;
    for (int pass = 0; pass < 4; ++pass) {
        if (wide)
            for (uint32_t it = threadIdx.x; it < n; it += blockDim.x) resolve_look<S>(d, it);
        // a warp per pending cell, lane q its neighbour in direction q
        for (uint32_t it = threadIdx.x >> 5; !wide && it < n; it += blockDim.x >> 5) {
            const int lane = threadIdx.x & 31;
            const long long i = d.list[WL_PEND][it];
            if (!(d.cmark[i] & MK_PEND)) {
                if (lane == 0) d.rdec[it] = 0;
                continue;
            }
            int x, y, z;
            coords(d, i, x, y, z);
            const long long yi = lane_nbr(d, lane, x, y, z);
            // mark, class, density and fill level of the neighbour requested
            // together (those of a cell without populations are not used)
            const int mk = yi < 0 ? MK_PEND : d.cmark[yi], cl = cls(d, yi), c = (mk & MK_PEND) ? 0 : cl;
            double r = 0.0, ph = 0.0;
            if (cl == CL_L || cl == CL_I) r = cell_density<S>(d, d.fdst, yi);
            if (cl == CL_I) ph = d.phidst[yi];
            const unsigned full = 0xffffffffu;
            const unsigned mL = __ballot_sync(full, c == CL_L), mI = __ballot_sync(full, c == CL_I),
                           mG = __ballot_sync(full, c == CL_G);
            const int nL = __popc(mL), nI = __popc(mI), nG = __popc(mG);
            // sums in q order
            double sr = 0.0, sp = 0.0;
            for (unsigned m = mL | mI; m; m &= m - 1) sr += __shfl_sync(full, r, __ffs(m) - 1);
            for (unsigned m = mI; m; m &= m - 1) sp += __shfl_sync(full, ph, __ffs(m) - 1);
            if (lane == 0) resolve_decide(d, it, nL, nI, nG, sr, sp);
        }
        if (threadIdx.x == 0) s_any = 0;
        __syncthreads();
        if (wide)
            for (uint32_t it = threadIdx.x; it < n; it += blockDim.x)
                if (!resolve_set<S>(d, it, pass == 3)) s_any = 1;
        for (uint32_t it = threadIdx.x >> 5; !wide && it < n; it += blockDim.x >> 5) {
            const int lane = threadIdx.x & 31;
            const long long i = d.list[WL_PEND][it];
            const bool open = d.cmark[i] & MK_PEND;
            __syncwarp();
            if (!open) continue;
            int dec = d.rdec[it];
            if (dec == 0 && pass == 3) dec = CL_G;
            if (dec == 0) {
                if (lane == 0) s_any = 1;
                continue;
            }
            const Body &b = d.bodies_new[d.bid[i]];
            if (lane == 0) {
                d.cmark[i] = MK_FRESH;
                set_cls(d, i, dec);
            }
            if (dec == CL_G) continue;
            int x, y, z;
            coords(d, i, x, y, z);
            if (lane == 0 && z > *d.ztop_wr + ZTOP_MARGIN) atomicOr(d.status, ST_TOP);
            double p[3] = {x + 0.5, y + 0.5, z + 0.5}, uw[3];
            body_velocity_at(d, b, p, uw);
            const double rho = d.rrho[it];
            warp_store_cell<S>(d, i, lane, feq_lane(lane, rho, uw));
            __syncwarp();
            const double dens = warp_density<S>(d, d.fdst, i);
            if (lane == 0) {
                if (dec == CL_I) set_mass<S>(d, i, d.rphi[it] * rho, dens);
                d.rrho[it] = dens;  // as stored, for what follows
            }
        }
        __syncthreads();
        if (!s_any) break;
        __syncthreads();
    }
    // closure: a new liquid cell next to gas becomes interface with phi = 1
    for (uint32_t it = threadIdx.x >> 5; it < n; it += blockDim.x >> 5) {
        const int lane = threadIdx.x & 31;
        const long long i = d.list[WL_PEND][it];
        if (!(d.cmark[i] & MK_FRESH) || clsv(d, i) != CL_L) continue;
        int x, y, z;
        coords(d, i, x, y, z);
        const bool gas = __any_sync(0xffffffffu, cls(d, lane_nbr(d, lane, x, y, z)) == CL_G);
        if (lane == 0) d.rdec[it] = gas ? 1 : 0;
    }
    __syncthreads();
    double acc = 0.0;
    for (uint32_t it = threadIdx.x; it < n; it += blockDim.x) {
        long long i = d.list[WL_PEND][it];
        if (!(d.cmark[i] & MK_FRESH)) continue;
        const int c = clsv(d, i);
        if (c == CL_L) {
            const double r = d.rrho[it];
            acc += r;
            if (d.rdec[it]) {
                set_cls(d, i, CL_I);
                d.m[i] = r;
                d.phidst[i] = 1.0;  // r / r
                if constexpr (S != 0) d.phifdst[i] = 1.0f;
            }
        } else if (c == CL_I) {
            acc += d.m[i];
        }
        d.cmark[i] = 0;
    }
    __shared__ double sh[32];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        d.ledger[LG_UNCOVERED] += t;
    }
}

// ------------------------------------------- conversions and remap in one launch
//
// What follows the collision in a step -- the conversions, then the obstacle
// remapping -- is eleven short phases, each of which needs the one before it
// complete everywhere.  As kernels of their own they cost 3 to 6 us each even
// with empty lists, more than the work of a small tank's step, so one launch
// runs them with a barrier in between, and leaves out the conversions' (the
// remap's) barriers when nothing converts (no cell is covered or left).
// Measured, us, sum of the ten kernels timed one by one and this launch: 64^3
// without bodies 53 and 5; 130x40x40 117 and 40; 385x190x127 143 and 55;
// 768x384x256 172 and 72.
//  - CLUSTER, for tanks up to TAIL_CLUSTER_CELLS per plane: short lists by the
//    first cluster of TAIL_CLUSTER blocks with the hardware's cluster barrier,
//    the launch's other blocks leave at once (which costs nothing measurable);
//    long ones, of a splashing tank, by all blocks that have started by then
//    (tail_team);
//  - else a cooperative grid with a barrier in global memory, for large tanks
//    (hundreds to thousands of conversions a step want all SMs).
constexpr int TAIL_CLUSTER = 8, TAIL_BLOCKS = 152;
// Clusters launched: one per 65536 cells, at most the 15 that are resident at
// once (a tank of 32^3 cells has no list worth more than one).
constexpr int TAIL_CLUSTERS = 15;
constexpr long long TAIL_CLUSTER_PER = 65536;
// (1024 threads of the cluster's blocks give its short lists a warp each; on the
// grid they only make the block barriers longer: 768x384x256 103 us against 89)
constexpr int tail_threads(bool cluster) { return cluster ? 1024 : 512; }
// Entries (conversions, cells covered and left) up to which the first cluster
// works alone.  Measured, us of this launch, alone and with all blocks: 170
// entries 39 and 49, 210 41 and 48, 440 (FP32) 48 and 52, 450 (FP64) 84 and 60,
// 460 61 and 55, 840 64 and 49, 2900 199 and 67, 10900 677 and 132 (as ten
// kernels, timed one by one: 204 and 287 for the last two).
#ifndef LBMFS_TAIL_SHORT
#define LBMFS_TAIL_SHORT 512
#endif
constexpr uint32_t TAIL_SHORT = LBMFS_TAIL_SHORT;

// poll limit of the waits in global memory: far beyond the time that blocks
// which are all running can be apart
constexpr unsigned BARRIER_POLLS = 1u << 24;
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Barrier of the phases: of the cluster, or through global memory of the vb.nx
// blocks that work on them.
__device__ __forceinline__ bool tail_barrier(const Dev &d, const VB &vb, bool cluster) {
    if (cluster) {
        // (the form without .aligned: the warps may arrive diverged)
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        return true;
    }
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned *count = d.status + 1, *turn = d.status + 2;
        unsigned now;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(turn) : "memory");
        __threadfence();
        bool ok = true;
        if (atomicAdd(count, 1u) == vb.nx - 1) {
            *count = 0;
            __threadfence();
            atomicAdd(turn, 1u);
        } else {
            unsigned seen = now, polls = 0;
            for (; seen == now && polls < BARRIER_POLLS; ++polls) seen = ld_acquire(turn);
            ok = seen != now;
            if (!ok) atomicOr(d.status, ST_TIMEOUT);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}
// The blocks of an ordinary launch that work on long lists together: those that
// have come by the time the first of them closes the list of names, a few us
// after it started.  They are all running, so they can wait for one another
// whatever else the GPU is doing; blocks that come later leave.  The names are
// in the step's own counters, which are zero when it starts.  Sets the block's
// number and the number of blocks; false: not one of them.
constexpr unsigned TEAM_CLOSED = 1u << 31, TEAM_JOIN_POLLS = 16;
__device__ __forceinline__ bool tail_team(const Dev &d, VB &vb) {
    __shared__ unsigned s_rank, s_team;
    if (threadIdx.x == 0) {
        unsigned *names = d.cnt + CN_TEAM_NAMES, *size = d.cnt + CN_TEAM_SIZE;
        const unsigned rank = atomicAdd(names, 1u);
        unsigned team = 0;
        if (rank == 0) {
            for (unsigned polls = 0; polls < TEAM_JOIN_POLLS && ld_acquire(names) < gridDim.x; ++polls) {}
            team = atomicOr(names, TEAM_CLOSED);
            atomicExch(size, team);
        } else if (!(rank & TEAM_CLOSED)) {
            for (unsigned polls = 0; team == 0 && polls < BARRIER_POLLS; ++polls) team = ld_acquire(size);
            if (team == 0) atomicOr(d.status, ST_TIMEOUT);
        }
        s_rank = rank;
        s_team = team;
    }
    __syncthreads();
    vb.x = s_rank;
    vb.nx = s_team;
    return s_team != 0;
}

__device__ __forceinline__ uint32_t tail_conversions(const Dev &d) { return wl_count(d, WL_FILLED) + wl_count(d, WL_EMPTIED); }
__device__ __forceinline__ uint32_t tail_moved(const Dev &d) {
    return d.nb > 0 ? wl_count(d, WL_COVER) + wl_count(d, WL_PEND) : 0u;
}
__device__ __forceinline__ uint32_t tail_items(const Dev &d) { return tail_conversions(d) + tail_moved(d); }

template <int S, bool CLUSTER>
__global__ void __launch_bounds__(tail_threads(CLUSTER)) k_tail(const __grid_constant__ Dev d) {
    VB vb = vb_own();
    if (CLUSTER && vb.x >= TAIL_CLUSTER) {
        // (one thread looks: the counters of all 120 blocks' threads queueing at
        // one address cost 3 us)
        if (!__syncthreads_or(threadIdx.x == 0 && tail_items(d) > TAIL_SHORT)) return;
    }
    if (vb.x == 0) {
        // for the next step: its counters (this step's previous ones), and the
        // slot its bulk pass records the fluid top in
        if (threadIdx.x < CN_COUNT) d.pcnt[threadIdx.x] = 0;
        if (threadIdx.x == 0) *d.ztop_rd = -1;
    }
    const uint32_t nconv = tail_conversions(d), nmoved = tail_moved(d);
    bool cluster = false;
    if (CLUSTER && nconv + nmoved <= TAIL_SHORT) {
        vb.nx = TAIL_CLUSTER;
        cluster = true;
    } else if (CLUSTER && !tail_team(d, vb)) {
        return;
    }
    if (nconv) {
        // new interface cells are marked (the two lists mark disjoint cells)
        conv_filled_body(d, vb);
        conv_emptied_body(d, vb);
        if (!tail_barrier(d, vb, cluster)) return;
        // their states; the converted cells' shares and who receives them
        // (from the classes before and the marks)
        conv_init_body<S>(d, vb);
        conv_claim_body<S>(d, vb);
        if (!tail_barrier(d, vb, cluster)) return;
        conv_flags_body(d, vb);
        conv_excess_body<S>(d, vb);
        if (!tail_barrier(d, vb, cluster)) return;
        conv_finish_body(d, vb, nmoved > 0 && d.nb > 1);
    }
    if (nmoved) {
        remap_apply_body<S>(d, vb);
        if (!tail_barrier(d, vb, cluster)) return;
        if (vb.x == 0) remap_resolve_body<S>(d, vb);
        if (!tail_barrier(d, vb, cluster)) return;
        nb_update_body(d, vb);
    }
}

// ------------------------------------------------------ reductions, output

// sum over liquid rho + interface m -> red[block]
template <int S>
__global__ void __launch_bounds__(256) k_mass_partial(Dev d) {
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < d.N; i += (long long)gridDim.x * blockDim.x) {
        const int fb = d.flags[i], c = fb & CL_MASK;
        if (c == CL_L) {
            // closed interface layer (Sec. 2.2): no liquid cell touches gas; the
            // neighbours' classes are requested with the populations, off the
            // grid faces by constant index offsets
            bool gas = false;
            if (fb & (FACE_X | FACE_YZ)) {
                int x, y, z;
                coords(d, i, x, y, z);
#pragma unroll 1
                for (int q = 1; q < Q; ++q) gas = gas || cls(d, nbr(d, x, y, z, dir_x(q), dir_y(q), dir_z(q))) == CL_G;
            } else {
                const long long sy = d.nx, sz = (long long)d.nx * d.ny;
                unsigned any = 0;
#pragma unroll
                for (int q = 1; q < Q; ++q) any |= d.flags[i + (cx(q) + cy(q) * sy + cz(q) * sz)];
                gas = any & CL_G;
            }
            acc += cell_density<S>(d, d.fsrc, i);
            if (gas) atomicOr(d.status, ST_LIQUID_GAS);
        } else if (c == CL_I) {
            acc += d.m[i];
        }
    }
    __shared__ double sh[8];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        d.red[blockIdx.x] = t;
    }
}

__global__ void k_mass_final(Dev d, int nblk) {
    // one warp, in a fixed order (a double addition takes 65 cycles: one thread's
    // chain over all blocks took 10 us)
    double t = 0.0;
    for (int k = threadIdx.x; k < nblk; k += 32) t += d.red[k];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
    if (threadIdx.x == 0) d.ledger[LG_MASS] = t;
}

template <int S>
__global__ void k_read_fields(Dev d, unsigned mask, uint8_t *flags, double *fill, double *mass, double *rho, double *vel,
                              double *f) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= d.N) return;
    int c = clsv(d, i);
    bool fluid = c == CL_L || c == CL_I;
    double u[3] = {0.0, 0.0, 0.0};
    double r = fluid ? cell_rho_u<S>(d, d.fsrc, i, u) : 0.0;
    if (flags) flags[i] = (uint8_t)c;
    if (fill) fill[i] = c == CL_L ? 1.0 : (c == CL_I ? d.phisrc[i] : 0.0);
    if (mass) mass[i] = c == CL_L ? r : (c == CL_I ? d.m[i] : 0.0);
    if (rho) rho[i] = r;
    if (vel) {
        vel[3 * i] = u[0];
        vel[3 * i + 1] = u[1];
        vel[3 * i + 2] = u[2];
    }
    if (f)
        for (int q = 0; q < Q; ++q) f[(long long)q * d.N + i] = fluid ? Sto<S>::ldf(d.fsrc, q, i, d.N) : 0.0;
}

// ------------------------------------------------------------ launchers

// ------------------------------------------------------ batched launches
//
// One launch serves all tanks of a TankSet: block b runs the table entries
// b, b + gridDim.x, ... (a persistent walk when the grid is smaller than the
// table), each as the block of its tank's own grid that the entry names, with
// the block size of the single-tank launch.  The per-cell work is the
// single-tank kernels' own code.
template <class K>
__global__ void __launch_bounds__(K::THREADS, K::MINB)
    k_batch(const __grid_constant__ TankSet ts, const Tile *__restrict__ table, unsigned n, int zb) {
    launch_dependents();  // (of these only the bulk kernel is launched so, behind the force kernel)
    for (unsigned t = blockIdx.x; t < n; t += gridDim.x) {
        const Tile e = table[t];
        const VB vb{e.x, e.y, e.z, e.nx, e.ny, e.nz, e.kind};
        K::run(ts.d[e.tank], vb, zb);
        // the next entry's body reuses this one's shared memory; bodies
        // without shared memory let a block's warps move on independently
        if constexpr (K::SMEM) __syncthreads();
    }
}

// The short kernels of a batch's step (counters, conversions, rigid bodies,
// remap): the descriptors come from memory instead of the parameter space, 32 KB
// of which cost every launch a few us, and each launch is a programmatic
// dependent of the one before it in the chain.
template <class K>
__global__ void __launch_bounds__(K::THREADS, K::MINB)
    k_batch_short(const TankSet *__restrict__ ts, const Tile *__restrict__ table, unsigned n) {
    launch_dependents();
    wait_for_launch();
    for (unsigned t = blockIdx.x; t < n; t += gridDim.x) {
        const Tile e = table[t];
        const VB vb{e.x, e.y, e.z, e.nx, e.ny, e.nz, e.kind};
        const Dev d = ts->d[e.tank];  // (the fields that the body uses)
        K::run(d, vb, 0);
        if constexpr (K::SMEM) __syncthreads();
    }
}

#define LBMFS_BATCH_BODY_SM(NAME, THR, MB, SM, ...)                                           \
    struct NAME {                                                                              \
        static constexpr int THREADS = THR, MINB = MB;                                         \
        static constexpr bool SMEM = SM;                                                       \
        static __device__ __forceinline__ void run(const Dev &d, const VB &vb, int zb) { __VA_ARGS__; } \
    };
#define LBMFS_BATCH_BODY(NAME, THR, MB, ...) LBMFS_BATCH_BODY_SM(NAME, THR, MB, false, __VA_ARGS__)
struct BkReset {
    static constexpr int THREADS = 32, MINB = 1;
    static constexpr bool SMEM = false;
    static __device__ __forceinline__ void run(const Dev &d, const VB &, int) {
        if (threadIdx.x < CN_COUNT) d.cnt[threadIdx.x] = 0;
    }
};
template <int S> LBMFS_BATCH_BODY_SM(BkForces, FORCE_THREADS_BATCH, S == 0 ? 4 : LBMFS_FORCE_MINB, true, forces_body<S, true>(d, vb))
// one instantiation per z-planes-per-tile choice (the column loop unrolled to it)
template <int S, int ZB>
LBMFS_BATCH_BODY(BkLiquid, BULK_THREADS, S == 0 ? 1 : LBMFS_BULK_MINB, (liquid_body<S, ZB>(d, vb, zb)))
// the batch's listed cells are spread over many more blocks: 4 resident per SM
// (128 registers) beat 1 there, not on the single tank
template <int S>
LBMFS_BATCH_BODY_SM(BkGeneral, GEN_THREADS, 4, true, if (vb.kind == 0) near_body<S, true>(d, vb); else faces_body<S>(d, vb))
template <int S> LBMFS_BATCH_BODY(BkInterface, 128, S == 0 ? 2 : LBMFS_IFACE_MINB, interface_body<S>(d, vb))
// (runs after the bulk kernel, which has read this step's fluid top: clears the
// slot that the next step records its own in)
LBMFS_BATCH_BODY(BkConvFilled, LIST_THREADS, 1, if (vb.x == 0 && threadIdx.x == 0) *d.ztop_rd = -1; conv_filled_body(d, vb))
LBMFS_BATCH_BODY(BkConvEmptied, LIST_THREADS, 1, conv_emptied_body(d, vb))
template <int S> LBMFS_BATCH_BODY(BkConvInit, LIST_THREADS, 1, conv_init_body<S>(d, vb))
LBMFS_BATCH_BODY(BkConvFlags, LIST_THREADS, 1, conv_flags_body(d, vb))
template <int S> LBMFS_BATCH_BODY(BkConvClaim, LIST_THREADS, 1, conv_claim_body<S>(d, vb))
template <int S> LBMFS_BATCH_BODY(BkConvExcess, LIST_THREADS, 1, conv_excess_body<S>(d, vb))
LBMFS_BATCH_BODY(BkConvFinish, LIST_THREADS, 1, conv_finish_body(d, vb, false))
LBMFS_BATCH_BODY(BkBodies, 32, 1, bodies_body(d, vb))
LBMFS_BATCH_BODY(BkRemapScan, SCAN_THREADS, 1, remap_scan_body(d, vb))
template <int S> LBMFS_BATCH_BODY(BkRemapApply, LIST_THREADS, 1, remap_apply_body<S>(d, vb))
template <int S> LBMFS_BATCH_BODY_SM(BkRemapResolve, REMAP_THREADS, 1, true, remap_resolve_body<S>(d, vb))
LBMFS_BATCH_BODY(BkNbUpdate, LIST_THREADS, 1, nb_update_body(d, vb))
#undef LBMFS_BATCH_BODY
#undef LBMFS_BATCH_BODY_SM

// launch k, with `early` as a programmatic dependent of the stream's last kernel
// (see launch_dependents)
template <class... P, class... A>
void launch(void (*k)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, bool early, A... args) {
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute a = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&c, k, P(args)...);
}
template <class K> void batch_short(const BatchLaunch &b, int sh, int block, cudaStream_t st, bool early) {
    const Shape &x = b.sh[sh];
    if (x.n) launch(k_batch_short<K>, dim3(x.grid), block, 0, st, early, b.dts, x.table, x.n);
}
template <class K> void batch_launch(const BatchLaunch &b, int sh, dim3 block, cudaStream_t st) {
    const Shape &x = b.sh[sh];
    if (x.n) k_batch<K><<<x.grid, block, 0, st>>>(*b.ts, x.table, x.n, b.zb);
}
// z-planes per block of the single-tank bulk kernel.  A thread steps its planes
// one after another, so blocks of 8 planes suit only grids whose blocks still
// fill the GPU several times over; on smaller ones a few threads would walk 8
// dependent cells while SMs idle.  Measured (bulk kernel, us at 8 / 4 / 2 / 1
// planes): 32^3 FP64 111 / 60 / 34 / 21, 96^3 FP64 308 / 304 / 304 / 288;
// 96x32x32 FP32 27 / 17 / 12 / 10, 128^3 FP32 42 / 39 / 39 / 49, 385x190x127 FP32
// 138 / 135 / 156 / 246, 512x256x170 FP32 284 / 292 / 571 / 863; the 768x384x256
// tank 2 % faster at 8 than at 4.
inline int bulk_planes(int storage, unsigned gx, int nz) {
    auto blocks = [&](int zb) { return (long long)gx * ((nz + zb - 1) / zb); };
    if (storage == 0) return 1;  // bound by the double unit: the most even spread
    if (blocks(8) >= 12000) return 8;
    if (blocks(4) >= 12000) return 4;
    return blocks(2) >= 2000 ? 2 : 1;
}

// largest xy-plane whose tail starts as clusters; with a larger one hundreds of
// conversions a step are the rule (calm wave tanks measured with both forms, us:
// 385x190 plane 55 as a cluster, 65 as a grid; 768x384 109 and 82; a tank whose
// lists are empty 5 and 8)
constexpr long long TAIL_CLUSTER_CELLS = 131072;

constexpr int STEP_SLOTS = 7, BATCH_SLOTS = 17;  // kernel slots of a step (names below)

template <int S> struct Launch {
    static void init_cells(const Dev &d, const uint8_t *flags, const double *fill, const double *rho, const double *vel,
                           cudaStream_t st) {
        unsigned blocks = (unsigned)((d.N + 255) / 256);
        k_init<S><<<blocks, 256, 0, st>>>(d, flags, fill, rho, vel);
        Dev prev = d;  // the lists of the step before the first
        prev.list[WL_IFACE] = const_cast<uint32_t *>(d.plist[0]);
        prev.cnt = d.pcnt;
        k_list_interface<<<blocks, 256, 0, st>>>(prev);
        k_nb_all<<<dim3((d.nx + 127) / 128, d.ny, d.nz), 128, 0, st>>>(d);
    }
    static void body_prepare(const Dev &d, int b, cudaStream_t st) { k_body_prepare<<<1, 32, 0, st>>>(d, b); }
    static void map_body(const Dev &d, int b, int book, cudaStream_t st) {
        k_map_body<S><<<FORCE_BLOCKS, 256, 0, st>>>(d, b, book);
        k_nb_body<<<FORCE_BLOCKS, dim3(32, 8), 0, st>>>(d, b);
    }
    static void liquid_mass(const Dev &d, cudaStream_t st) {
        k_mass_partial<S><<<LIST_BLOCKS, 256, 0, st>>>(d);
        k_mass_final<<<1, 32, 0, st>>>(d, LIST_BLOCKS);
    }
    static void read_fields(const Dev &d, unsigned mask, void *const *dst, cudaStream_t st) {
        unsigned blocks = (unsigned)((d.N + 255) / 256);
        k_read_fields<S><<<blocks, 256, 0, st>>>(
            d, mask, (mask & 1u) ? (uint8_t *)dst[0] : nullptr, (mask & 2u) ? (double *)dst[1] : nullptr,
            (mask & 4u) ? (double *)dst[2] : nullptr, (mask & 8u) ? (double *)dst[3] : nullptr,
            (mask & 16u) ? (double *)dst[4] : nullptr, (mask & 32u) ? (double *)dst[5] : nullptr);
    }
    static void faces(const Dev &d, cudaStream_t st) { k_faces<S><<<LIST_BLOCKS, GEN_THREADS, 0, st>>>(d); }
    static void near(const Dev &d, cudaStream_t st) {
        k_near<S><<<d.loose ? dim3(4 * LIST_BLOCKS) : dim3(d.range_blocks, d.nb), GEN_THREADS, 0, st>>>(d);
    }
    static void forces(const Dev &d, cudaStream_t st) {
        k_forces<S><<<dim3(FORCE_BLOCKS, d.nb), FORCE_THREADS, 0, st>>>(d);
    }
    static void scan(const Dev &d, cudaStream_t st, bool early) {
        // a cell or two per thread; blocks small enough to run beside the ring
        // kernel's, which leave 4096 registers of an SM
        launch(k_remap_scan, dim3(std::max(d.range_blocks, 1216 / d.nb), d.nb), SCAN_THREADS, 0, st, early, d);
    }
    static void interface(const Dev &d, cudaStream_t st) { k_interface<S><<<LBMFS_IFACE_GRID, 128, 0, st>>>(d); }
    // the bulk kernel: FP64 and FP32 one cell per thread, with the z-planes per
    // block of bulk_planes; FP16 the ring, or on narrow grids one cell per thread
    // and a plane per block; LBMFS_BULK selects the staged forms
    static void bulk_any(const Dev &d, cudaStream_t st, bool early) {
        if constexpr (S != 0) {
            // the staged variants tile rows: (ceil(nx / BULK_THREADS), ny, z-blocks)
            dim3 rgrid((d.nx + BULK_THREADS - 1) / BULK_THREADS, d.ny, (d.nz + LBMFS_BULK_ZB - 1) / LBMFS_BULK_ZB);
            dim3 pgrid(rgrid.x, rgrid.y, (d.nz + LBMFS_BULK_PIPE_ZB - 1) / LBMFS_BULK_PIPE_ZB);
            if (d.bulk == BULK_TMA) {
                k_liquid_tma<S><<<rgrid, BULK_THREADS, 128 + 2 * Stage<S>::BYTES, st>>>(d);
                return;
            }
            if (d.bulk == BULK_PIPE) {
                k_liquid_pipe<S><<<pgrid, BULK_THREADS, 0, st>>>(d);
                return;
            }
        }
        if (S == 2 && d.nx >= RING_MIN_NX) {
            using G = RingShape;
            const uint32_t n = (uint32_t)((d.N + G::TILE - 1) / G::TILE);
            const auto k = d.a_f[0] == 0.0f && d.a_f[1] == 0.0f ? k_ring<true> : k_ring<false>;
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
            launch(k, dim3(std::min(n, 152u * RING_CTAS)), G::THREADS, G::SMEM, st, early, d, n);
        } else {
            const unsigned gx = (unsigned)(((long long)d.nx * d.ny + BULK_THREADS - 1) / BULK_THREADS);
            const int zb = S == 2 ? 1 : bulk_planes(S, gx, d.nz);
            auto go = [&](void (*k)(Dev)) { launch(k, dim3(gx, 1, (d.nz + zb - 1) / zb), BULK_THREADS, 0, st, early, d); };
            if (zb == 1) go(k_liquid<S, 1>);
            if constexpr (S == 1) {
                if (zb == 2) go(k_liquid<S, 2>);
                if (zb == 4) go(k_liquid<S, 4>);
                if (zb == 8) go(k_liquid<S, 8>);
            }
        }
    }
    static void tail(const Dev &d, cudaStream_t st) {
        cudaLaunchConfig_t c = {};
        cudaLaunchAttribute a = {};
        c.stream = st;
        c.attrs = &a;
        c.numAttrs = 1;
        if ((long long)d.nx * d.ny <= TAIL_CLUSTER_CELLS) {
            c.gridDim = dim3(TAIL_CLUSTER * std::max(1, (int)std::min<long long>(TAIL_CLUSTERS, d.N / TAIL_CLUSTER_PER)));
            c.blockDim = dim3(tail_threads(true));
            a.id = cudaLaunchAttributeClusterDimension;
            a.val.clusterDim.x = TAIL_CLUSTER;
            a.val.clusterDim.y = a.val.clusterDim.z = 1;
            cudaLaunchKernelEx(&c, k_tail<S, true>, d);
        } else {
            // a block per SM, of the SMs that there are (all blocks are resident)
            int dev = 0, sms = TAIL_BLOCKS;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            c.gridDim = dim3(std::min(TAIL_BLOCKS, sms));
            c.blockDim = dim3(tail_threads(false));
            a.id = cudaLaunchAttributeCooperative;
            a.val.cooperative = 1;
            cudaLaunchKernelEx(&c, k_tail<S, false>, d);
        }
    }
    // One time step.  The force kernel, the rigid-body update and the remap's
    // scan (a chain), the cells next to bodies or on moving walls, and the
    // interface cells need only the state at t: with `sides` (while a graph is
    // captured) these chains run beside the bulk kernel, on streams of a higher
    // priority, and join before the tail; the bulk kernel is launched behind the
    // start of the force kernel, the first of the longest chain
    // (launch_dependents).  Without, all run in one chain.  With
    // ev != nullptr event k is recorded before kernel slot k (step_names).
    static int step(const Dev &d, cudaStream_t st, const Sides *sides, cudaEvent_t *ev) {
        const bool bodies = d.nb > 0, obstacles = bodies || d.loose, walls = d.walls_move != 0;
        const int launches = 3 + (bodies ? 3 : 0) + (obstacles ? 1 : 0) + (walls ? 1 : 0);
        if (sides) {
            const bool used[SIDE_STREAMS] = {true, bodies, obstacles || walls};
            cudaEventRecord(sides->fork, st);
            for (int k = 0; k < SIDE_STREAMS; k += 2)
                if (used[k]) cudaStreamWaitEvent(sides->st[k], sides->fork, 0);
            if (bodies) {
                forces(d, st);
                cudaEventRecord(sides->fork2, st);
                cudaStreamWaitEvent(sides->st[1], sides->fork2, 0);
            }
            if (obstacles) near(d, sides->st[2]);
            if (walls) faces(d, sides->st[2]);
            interface(d, sides->st[0]);
            if (bodies) launch_bodies(d, sides->st[1]);
            if (bodies) scan(d, sides->st[1], true);
            bulk_any(d, st, bodies);  // (behind the force kernel's start)
            for (int k = 0; k < SIDE_STREAMS; ++k)
                if (used[k]) {
                    cudaEventRecord(sides->join[k], sides->st[k]);
                    cudaStreamWaitEvent(st, sides->join[k], 0);
                }
            tail(d, st);
            return launches;
        }
        int k = 0;
        auto mark = [&]() {
            if (ev) cudaEventRecord(ev[k], st);
            ++k;
        };
        mark();
        if (bodies) forces(d, st);
        mark();
        bulk_any(d, st, false);
        mark();
        if (obstacles) near(d, st);
        if (walls) faces(d, st);
        mark();
        interface(d, st);
        mark();
        if (bodies) launch_bodies(d, st);
        mark();
        if (bodies) scan(d, st, false);
        mark();
        tail(d, st);
        mark();
        return launches;
    }
};

// (early: behind the start of the stream's last kernel, see launch_dependents)
template <int S> void batch_bulk_launch(const BatchLaunch &b, cudaStream_t st, bool early) {
    const Shape &x = b.sh[SH_BULK];
    if constexpr (S == 2) {
        const Shape &narrow = b.sh[SH_NARROW];
        if (narrow.n)
            launch(k_batch<BkLiquid<S, 1>>, dim3(narrow.grid), BULK_THREADS, 0, st, early, *b.ts, narrow.table, narrow.n, 1);
        if (!x.n) return;
        const auto k = b.zg ? k_batch_ring<true> : k_batch_ring<false>;
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RingShape::SMEM);
        launch(k, dim3(x.grid), RingShape::THREADS, RingShape::SMEM, st, early && !narrow.n, *b.ts, x.table, x.n);
    } else {
        auto go = [&](void (*k)(TankSet, const Tile *, unsigned, int)) {
            launch(k, dim3(x.grid), BULK_THREADS, 0, st, early, *b.ts, x.table, x.n, b.zb);
        };
        if (b.zb == 1) go(k_batch<BkLiquid<S, 1>>);
        else if (b.zb == 2) go(k_batch<BkLiquid<S, 2>>);
        else if (b.zb == 4) go(k_batch<BkLiquid<S, 4>>);
        else go(k_batch<BkLiquid<S, 8>>);
    }
}

// The batched counterpart of Launch<S>::step (same kernel slots).
template <int S> struct BatchStep {
    // (with sides: the chains that need only the state at t beside the bulk
    // kernel, as in Launch<S>::step)
    static int step(const BatchLaunch &b, cudaStream_t st, const Sides *sides, cudaEvent_t *ev) {
        int k = 0;
        auto mark = [&]() {
            if (ev) cudaEventRecord(ev[k], st);
            ++k;
        };
        mark();
        const bool chain = ev == nullptr;  // (an event between two launches breaks the chain)
        batch_short<BkReset>(b, SH_TANK, 32, st, false);
        cudaStream_t s0 = st, s1 = st, s2 = st;
        if (sides) {
            cudaEventRecord(sides->fork, st);
            for (int j = 0; j < SIDE_STREAMS; j += 2) cudaStreamWaitEvent(sides->st[j], sides->fork, 0);
            s0 = sides->st[0];
            s1 = sides->st[1];
            s2 = sides->st[2];
        }
        mark();
        batch_launch<BkForces<S>>(b, SH_FORCE, FORCE_THREADS_BATCH, st);
        if (sides) {
            cudaEventRecord(sides->fork2, st);
            cudaStreamWaitEvent(s1, sides->fork2, 0);
            batch_launch<BkGeneral<S>>(b, SH_GEN, GEN_THREADS, s2);
            batch_launch<BkInterface<S>>(b, SH_IFACE, 128, s0);
            launch_bodies_batch(b, s1, false);
            batch_short<BkRemapScan>(b, SH_SCAN, SCAN_THREADS, s1, true);
        }
        mark();
        batch_bulk_launch<S>(b, st, sides != nullptr && b.sh[SH_FORCE].n > 0);
        mark();
        if (!sides) batch_launch<BkGeneral<S>>(b, SH_GEN, GEN_THREADS, s2);
        mark();
        if (!sides) batch_launch<BkInterface<S>>(b, SH_IFACE, 128, st);
        mark();
        if (sides)
            for (int j = 0; j < SIDE_STREAMS; ++j) {
                cudaEventRecord(sides->join[j], sides->st[j]);
                cudaStreamWaitEvent(st, sides->join[j], 0);
            }
        batch_short<BkConvFilled>(b, SH_LIST, LIST_THREADS, st, false);
        mark();
        batch_short<BkConvEmptied>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkConvInit<S>>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkConvClaim<S>>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkConvFlags>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkConvExcess<S>>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkConvFinish>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        if (!sides) launch_bodies_batch(b, st, false);
        mark();
        if (!sides) batch_short<BkRemapScan>(b, SH_SCAN, SCAN_THREADS, st, false);
        mark();
        batch_short<BkRemapApply<S>>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        batch_short<BkRemapResolve<S>>(b, SH_ONE, REMAP_THREADS, st, chain);
        mark();
        batch_short<BkNbUpdate>(b, SH_LIST, LIST_THREADS, st, chain);
        mark();
        int n = 0;
        const int shapes[] = {SH_TANK, SH_FORCE, SH_BULK, SH_NARROW, SH_GEN, SH_IFACE, SH_LIST, SH_LIST, SH_LIST, SH_LIST,
                              SH_LIST, SH_LIST, SH_LIST, SH_BODY, SH_SCAN, SH_LIST, SH_ONE, SH_LIST};
        for (int sh : shapes) n += b.sh[sh].n ? 1 : 0;
        return n;
    }
    static void bulk(const BatchLaunch &b, cudaStream_t st) { batch_bulk_launch<S>(b, st, false); }
    static int bulk_blocks_per_sm() {
        int nb = 0;
        if constexpr (S == 2) nb = RING_CTAS;
        else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch<BkLiquid<S, 4>>, BULK_THREADS, 0) != cudaSuccess)
            return 1;
        return nb > 0 ? nb : 1;
    }
};

inline const char *const *step_names() {
    static const char *const n[] = {"forces", "liquid", "general", "interface", "bodies", "remap_scan", "convert_remap"};
    static_assert(sizeof n / sizeof n[0] == STEP_SLOTS, "one name per slot");
    return n;
}
inline const char *const *batch_names() {
    static const char *const n[] = {"reset_counters", "forces",     "liquid",     "general",     "interface",   "conv_filled",
                                    "conv_emptied",   "conv_init",  "conv_claim", "conv_flags",  "conv_excess", "conv_finish",
                                    "bodies",         "remap_scan", "remap_apply", "remap_resolve", "nb_update"};
    static_assert(sizeof n / sizeof n[0] == BATCH_SLOTS, "one name per slot");
    return n;
}

template <int S> KernelSet make_kernel_set() {
    KernelSet k;
    k.init_cells = &Launch<S>::init_cells;
    k.body_prepare = &Launch<S>::body_prepare;
    k.map_body = &Launch<S>::map_body;
    k.step = &Launch<S>::step;
    k.liquid_mass = &Launch<S>::liquid_mass;
    k.read_fields = &Launch<S>::read_fields;
    k.batch_step = &BatchStep<S>::step;
    k.batch_bulk = &BatchStep<S>::bulk;
    k.bulk_blocks_per_sm = &BatchStep<S>::bulk_blocks_per_sm;
    k.nkernels = STEP_SLOTS;
    k.names = step_names();
    k.batch_kernels = BATCH_SLOTS;
    k.batch_names = batch_names();
    return k;
}

}  // namespace
}  // namespace lbmfs
