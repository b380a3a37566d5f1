// wave.cuh -- K fused steps per launch for D2Q5 and D2Q9 as a row wavefront inside one warp.
//
// A warp owns a vertical strip of 64 columns (32 lanes x 2 consecutive columns, of which the
// outermost halo(K) on each side are recomputed) and a chunk of H output rows, which it
// sweeps upward.  In iteration r
//   level 0       takes row r of h^{t-1} (the stored post-collision populations),
//   level l >= 1  pulls, collides and hands on row r - l from level l - 1,
// so every level trails the one below by a row.  Of what a site of level l pulls from
// level l - 1 (Eq. BGK-LB lhs, g_i(x, t) = h_i(x - c_i, t - 1)) the populations with
// c_y = -1 were computed just before in this iteration, those with c_y = 0 in the previous one
// and those with c_y = +1 two iterations back; all of them sit in the lane's registers.  The
// x shifts take one shuffle per population.  Nothing is shared between warps: no barrier.
//
// What bounds it and why this shape: the one-step kernel is bound by HBM (41 B per D2Q5 site
// and step), and K fused steps move 41 / K; what is left is the latency of two to three warps per
// scheduler, which fill 50 % (BF16: 67 %) of the issue slots.  A CTA-wide wavefront (256 columns, one a thread, x neighbours through shared memory
// and a barrier per row) took 74 instructions per site and step and reached 316 GLUPS.  Here two
// columns per lane go through packed FP32 operations (f32x2), neighbours come by shuffle, and
// an iteration of four levels is about 225 instructions for 56 x 4 site updates.  Four columns
// per lane needed 168 registers and twice the code: it spilled and starved on instruction
// fetch (190 GLUPS where two columns gave 340).  GB300, 4096^2 / 8192^2, us a step before and
// after: D2Q5 FP32 100.5 -> 30.1 / 398 -> 100 (K = 6), BF16 60.6 -> 29.6 / 256 -> 103 (K = 4),
// MRT FP32 100.6 -> 32.0, D2Q9 FP32 184 -> 63.6 (K = 4).
//
// Rows arrive by cp.async in a ring of kRing row slots per warp, kRing - 1 rows ahead, and
// each lane reads only what it copied itself.  A second ring keeps the medium and the sponge
// factor of the last K + 1 rows, formed once per row.
//
// The arithmetic of a site is that of the one-step kernels, operation by operation, and
// 16-bit storage is rounded after every level (ROUND), so a fused launch gives the one-step
// kernels' results bit for bit.
#pragma once

#include <cuda_runtime.h>

#include "lb_kernels.cuh"

namespace lbwave {

using namespace lbk;

constexpr int kWarpsPerCta = 4;
constexpr int kCtaThreads = 32 * kWarpsPerCta;
constexpr int kCols = 64;   // columns of a strip
constexpr int kRing = 3;    // row slots per warp
constexpr int kMedRow = 32 * 16;  // bytes of a row in the medium ring: per lane m, m, f, f

enum { kLossless = 0, kBgk = 1, kMrt = 2 };  // D2Q5 BGK with omega = 2; BGK; MRT
enum { kZeroGhost = 0, kPeriodic = 1, kEither = 2 };  // a kernel's boundary (kEither: WaveArgs::per)

// recomputed columns on each side: K rounded up to whole lanes
__host__ __device__ constexpr int halo(int K) { return (K + 1) / 2 * 2; }
__host__ __device__ constexpr int out_cols(int K) { return kCols - 2 * halo(K); }
// rows of the medium ring: a power of two above K + 1 (the spare row passes receiver pressures)
__host__ __device__ constexpr int med_rows(int K) { return K < 3 ? 4 : K < 7 ? 8 : 16; }

template <int Q, typename ST> __host__ __device__ constexpr int slot_bytes() {
    return Q * kCols * (int)sizeof(ST) + kCols * 4;
}
template <int Q, int K, typename ST> __host__ __device__ constexpr int warp_bytes() {
    return kRing * slot_bytes<Q, ST>() + med_rows(K) * kMedRow;
}
template <int Q, int K, typename ST> __host__ __device__ constexpr int cta_bytes() {
    return kWarpsPerCta * warp_bytes<Q, K, ST>() + 256 * 4;
}

struct WaveArgs {
    const int *row_off;  // [ny + 1]: the receivers of row y are entries row_off[y] .. row_off[y+1]
    const int *rec_x;    // their x, ascending within a row
    const int *rec_y;    // their row
    const int *rec_id;   // their receiver index
    int strips;          // warps along x, of which the first edge_l and the last edge_r meet
    int edge_l, edge_r;  // the sponge or a zero-ghost face
    int chunks, chunks_e;  // row chunks of the others and of those
    int outer;           // what a row in the sponge counts (chunk_row)
    int tasks;           // warps with work
    int per;             // periodic boundary
    int bf16;            // served batches: the shot's storage is BF16 (else FP32)
};

// First row of chunk k of n.  Rows in the sponge count `outer` and the others kInner, as their
// iterations take, and every chunk gets the same sum (a strip in the x sponge counts all its
// rows alike: uniform).
constexpr int kInner = 6;
__host__ __device__ __forceinline__ int chunk_row(int k, int n, int ny, int sponge, int outer,
                                                  bool uniform) {
    if (uniform) return (int)((long long)ny * k / n);
    const long long w = sponge < ny / 2 ? sponge : ny / 2, mid = kInner * (ny - 2 * w);
    const long long c = (2 * outer * w + mid) * k / n;
    if (c <= outer * w) return (int)(c / outer);
    if (c <= outer * w + mid) return (int)(w + (c - outer * w) / kInner);
    return (int)(ny - w + (c - outer * w - mid) / outer);
}

// wrap_mod for values mostly within one period of the grid
__device__ __forceinline__ int wrap1(int v, int n) {
    if (v < 0) v += n;
    if (v >= n) v -= n;
    return (unsigned)v < (unsigned)n ? v : wrap_mod(v, n);
}

// ------------------------------------------------------------------ row copies --
template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src, bool live) {
    const int n = live ? BYTES : 0;  // 0: the destination is filled with zeros
    asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(n),
                 "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ float2 lds2(uint32_t at) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(at));
    return v;
}
__device__ __forceinline__ uint32_t lds1(uint32_t at) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at));
    return v;
}

// ------------------------------------------------------- two columns of a lane --
// Blackwell's packed FP32 operations (add / mul / fma .rn.f32x2) take one instruction for two
// columns and round each as the scalar operation does.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma(float a, float2 b, float2 c) { return __ffma2_rn(f2(a), b, c); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return fma(-1.f, b, a); }

// their form in memory
template <typename ST> struct Two;
template <> struct Two<float> {
    __device__ static __forceinline__ float2 lds(uint32_t at) { return lds2(at); }
    __device__ static __forceinline__ void store(float *o, float2 v) {
        *reinterpret_cast<float2 *>(o) = v;
    }
    __device__ static __forceinline__ float2 round(float2 v) { return v; }
};
template <> struct Two<__nv_bfloat16> {
    __device__ static __forceinline__ uint32_t pack(float2 a) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a.x, a.y);
        return *reinterpret_cast<const uint32_t *>(&h);
    }
    __device__ static __forceinline__ float2 unpack(uint32_t u) {
        return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
    }
    __device__ static __forceinline__ float2 lds(uint32_t at) { return unpack(lds1(at)); }
    __device__ static __forceinline__ void store(__nv_bfloat16 *o, float2 v) {
        *reinterpret_cast<uint32_t *>(o) = pack(v);
    }
    // the values a store and a load would give
    __device__ static __forceinline__ float2 round(float2 v) { return unpack(pack(v)); }
};

template <> struct Two<__half> {
    __device__ static __forceinline__ uint32_t pack(float2 a) {
        const __half2 h = __floats2half2_rn(a.x, a.y);
        return *reinterpret_cast<const uint32_t *>(&h);
    }
    __device__ static __forceinline__ float2 unpack(uint32_t u) {
        return __half22float2(*reinterpret_cast<const __half2 *>(&u));
    }
    __device__ static __forceinline__ float2 lds(uint32_t at) { return unpack(lds1(at)); }
    __device__ static __forceinline__ void store(__half *o, float2 v) {
        *reinterpret_cast<uint32_t *>(o) = pack(v);
    }
    __device__ static __forceinline__ float2 round(float2 v) { return unpack(pack(v)); }
};

// FP16's range scales (StepArgs): of the input, of the first step's values and of the output, and
// the largest values of both steps.  The other types have none.
template <int Q, typename ST> struct Range {
    __device__ __forceinline__ explicit Range(const StepArgs &) {}
    __device__ __forceinline__ float2 input(int, float2 v) const { return v; }
    __device__ __forceinline__ float2 between(int, float2 v, bool) { return Two<ST>::round(v); }
    __device__ __forceinline__ float2 output(int, float2 v) { return v; }
    __device__ __forceinline__ void fold(const StepArgs &, int, bool) const {}
};
template <int Q> struct Range<Q, __half> {
    float in[Q], mid[Q], imid[Q], out[Q], top1[Q], top2[Q];
    __device__ __forceinline__ explicit Range(const StepArgs &a) {
#pragma unroll
        for (int i = 0; i < Q; i++) {
            in[i] = a.scale_in[i];
            mid[i] = a.scale_out[i];
            imid[i] = 1.f / mid[i];  // exact: powers of two
            out[i] = 1.f / a.scale_two[i];
            top1[i] = top2[i] = 0.f;
        }
    }
    __device__ __forceinline__ float2 input(int i, float2 v) const { return mul(f2(in[i]), v); }
    // row: one of the chunk's own (warp-uniform)
    __device__ __forceinline__ float2 between(int i, float2 v, bool row) {
        if (row) top1[i] = fmaxf(top1[i], fmaxf(fabsf(v.x), fabsf(v.y)));
        return mul(f2(mid[i]), Two<__half>::round(mul(f2(imid[i]), v)));
    }
    __device__ __forceinline__ float2 output(int i, float2 v) {
        top2[i] = fmaxf(top2[i], fmaxf(fabsf(v.x), fabsf(v.y)));
        return mul(f2(out[i]), v);
    }
    // every lane of the warp; own: its columns are output columns
    __device__ __forceinline__ void fold(const StepArgs &a, int lane, bool own) const {
#pragma unroll
        for (int i = 0; i < Q; i++) {  // non-negative floats order as their bits
            const unsigned m1 = __reduce_max_sync(0xffffffffu, own ? __float_as_uint(top1[i]) : 0u);
            const unsigned m2 = __reduce_max_sync(0xffffffffu, own ? __float_as_uint(top2[i]) : 0u);
            const int at = i * kMaxCopies + blockIdx.x % kMaxCopies;
            if (lane == 0) {
                atomicMax(a.max_out + at, m1);
                atomicMax(a.max_two + at, m2);
            }
        }
    }
};

// Nothing crosses a face of a zero-ghost grid.  Sites beyond it are computed too and multiplied by 0,
// but that keeps a non-finite value, which the one-step kernels lose across the face.  So what
// leaves the first column to the left and the last to the right is set to 0.
__device__ __forceinline__ void cut_left(float2 &h, int gx) { h.x = gx == 0 ? 0.f : h.x; }
__device__ __forceinline__ void cut_right(float2 &h, int gx, int nx) {
    h.x = gx == nx - 1 ? 0.f : h.x;
    h.y = gx == nx - 2 ? 0.f : h.y;
}

// the values at x - 1 and x + 1 of a lane's columns
__device__ __forceinline__ float2 from_left(float2 h) {
    return make_float2(__shfl_up_sync(0xffffffffu, h.y, 1), h.x);
}
__device__ __forceinline__ float2 from_right(float2 h) {
    return make_float2(h.y, __shfl_down_sync(0xffffffffu, h.x, 1));
}

// ------------------------------------------------------------------- collision --
// m: w_1 = eta^2 / 4 for D2Q5 (formed once per row), eta^2 for D2Q9
template <int Q> __device__ __forceinline__ float med_of(float e2) { return Q == 5 ? 0.25f * e2 : e2; }
template <int Q> __device__ __forceinline__ float e2_of(float m) { return Q == 5 ? 4.f * m : m; }  // exact

// The lossless form hands on -h in place of h: g* = 2 g^eq - g is one fused multiply-add per
// population as -g* = g - 2 g^eq, and rounding to nearest is symmetric, so the next level
// works on the negated values throughout and restores the sign.  Level l's values carry
// sign<CK>(l); an even number of levels ends on the plain sign.
template <int CK> __device__ __forceinline__ constexpr float sign(int l) {
    return CK == kLossless && (l & 1) ? -1.f : 1.f;
}

// in place: g becomes h (lossless: -h)
template <int Q, int CK>
__device__ __forceinline__ void collide(float2 (&g)[Q], float2 m, const StepArgs &a) {
    if constexpr (Q == 5 && CK != kMrt) {
        const float2 rho = add(add(add(add(g[0], g[1]), g[2]), g[3]), g[4]);
        const float2 jx = sub(g[1], g[3]), jy = sub(g[2], g[4]);
        const float2 b = mul(m, rho), eq0 = fma(-4.f, b, rho);
        const float2 eq1 = fma(0.5f, jx, b), eq3 = fma(-0.5f, jx, b);
        const float2 eq2 = fma(0.5f, jy, b), eq4 = fma(-0.5f, jy, b);
        if constexpr (CK == kLossless) {  // collide5_lossless, operation by operation
            g[0] = fma(-2.f, eq0, g[0]);
            g[1] = fma(-2.f, eq1, g[1]);
            g[2] = fma(-2.f, eq2, g[2]);
            g[3] = fma(-2.f, eq3, g[3]);
            g[4] = fma(-2.f, eq4, g[4]);
        } else {  // collide5<false>
            const float om = a.omega;
            g[0] = fma(om, sub(eq0, g[0]), g[0]);
            g[1] = fma(om, sub(eq1, g[1]), g[1]);
            g[2] = fma(om, sub(eq2, g[2]), g[2]);
            g[3] = fma(om, sub(eq3, g[3]), g[3]);
            g[4] = fma(om, sub(eq4, g[4]), g[4]);
        }
    } else if constexpr (Q == 5) {  // collide5<true>, with the fused operations it compiles to
        const float2 rho = add(add(add(add(g[0], g[1]), g[2]), g[3]), g[4]);
        const float2 c = fma(-20.f, m, f2(4.f));  // 4 - 5 eta^2
        const float2 de = mul(f2(a.s[3]), fma2(c, rho, fma(-5.f, g[0], rho)));
        const float2 pxx = sub(add(sub(g[1], g[2]), g[3]), g[4]);
        const float2 sum = fma(a.s[4], pxx, de), dif = fma(-a.s[4], pxx, de);
        g[0] = fma(4.f, de, g[0]);
        g[1] = sub(g[1], sum);
        g[2] = sub(g[2], dif);
        g[3] = sub(g[3], sum);
        g[4] = sub(g[4], dif);
    } else if constexpr (CK != kMrt) {  // collide9<false>, with the fused operations it compiles to
        float2 rho = g[0];
#pragma unroll
        for (int i = 1; i < 9; i++) rho = add(rho, g[i]);
        const float2 jx = add(sub(sub(add(sub(g[1], g[3]), g[5]), g[6]), g[7]), g[8]);
        const float2 jy = sub(sub(add(add(sub(g[2], g[4]), g[5]), g[6]), g[7]), g[8]);
        const float2 w1 = mul(m, f2(a.w1r)), b1 = mul(w1, rho), b5 = mul(mul(m, f2(a.w5r)), rho);
        const float2 eq0 = fma(-4.f, fma2(w1, rho, b5), rho), sp = add(jx, jy), sm = sub(jx, jy);
        const float om = a.omega;
        auto relax = [om](float2 eq, float2 h) { return fma(om, sub(eq, h), h); };
        g[0] = relax(eq0, g[0]);
        g[1] = relax(fma(a.a1, jx, b1), g[1]);
        g[2] = relax(fma(a.a1, jy, b1), g[2]);
        g[3] = relax(fma(-a.a1, jx, b1), g[3]);
        g[4] = relax(fma(-a.a1, jy, b1), g[4]);
        g[5] = relax(fma(a.a5, sp, b5), g[5]);
        g[6] = relax(fma(-a.a5, sm, b5), g[6]);
        g[7] = relax(fma(-a.a5, sp, b5), g[7]);
        g[8] = relax(fma(a.a5, sm, b5), g[8]);
    } else {  // collide9<true>, with the fused operations it compiles to
        const float2 A = add(g[1], g[3]), B = add(g[2], g[4]), C = add(g[5], g[7]), D = add(g[6], g[8]);
        const float2 s14 = add(A, B), s58 = add(C, D), re2 = mul(add(add(g[0], s14), s58), m);
        const float c3 = 12.f * a.w1r + 24.f * a.w5r, c5 = 24.f * a.w1r + 12.f * a.w5r;
        const float kq = 4.f * (a.a5 - a.a1), ka = -2.f - kq, kb = 1.f - kq;
        const float2 X1 = sub(g[1], g[3]), Y1 = sub(g[2], g[4]);
        const float2 u = sub(g[5], g[7]), v = sub(g[6], g[8]), X5 = sub(u, v), Y5 = add(u, v);
        const float2 d3 = mul(f2(a.s[3]), fma(-c3, re2, fma(3.f, s14, mul(f2(6.f), s58))));
        const float2 d5 = mul(f2(a.s[5]), fma(-3.f, s58, fma(c5, re2, mul(f2(-6.f), s14))));
        const float2 d6 = mul(f2(a.s[6]), fma(ka, X1, mul(f2(kb), X5)));
        const float2 d7 = mul(f2(a.s[7]), fma(ka, Y1, mul(f2(kb), Y5)));
        const float2 x4 = sub(A, B), x8 = sub(C, D), n3 = mul(f2(-1.f), d3);
        g[0] = sub(g[0], fma(4.f, d5, mul(f2(-4.f), d3)));
        const float2 p = fma(-2.f, d5, fma(a.s[4], x4, n3)), q = fma(-2.f, d5, fma(-a.s[4], x4, n3));
        g[1] = sub(g[1], fma(-2.f, d6, p));
        g[2] = sub(g[2], fma(-2.f, d7, q));
        g[3] = sub(g[3], fma(2.f, d6, p));
        g[4] = sub(g[4], fma(2.f, d7, q));
        const float2 cc = fma(2.f, d3, d5), e = add(cc, d6), f = sub(cc, d6);
        g[5] = sub(g[5], fma(a.s[8], x8, add(e, d7)));
        g[6] = sub(g[6], fma(-a.s[8], x8, add(f, d7)));
        g[7] = sub(g[7], fma(a.s[8], x8, sub(f, d7)));
        g[8] = sub(g[8], fma(-a.s[8], x8, sub(e, d7)));
    }
}

// ------------------------------------------------------------------------ warp --
// Per-lane constants of one strip and row chunk.
struct Lane {
    int lane, gx, gxw;     // first column, and its periodic image
    int Y0, Y1;
    int own0, own1;        // the strip's output columns inside the grid, from its first column
    bool per, own;         // own: the lane's columns are output columns inside the grid
    bool live;             // zero ghost: some column inside the grid
    bool split;            // periodic: the two columns are not one aligned vector in memory
    bool src;              // warp-uniform: the source column is among the strip's
    bool face;             // warp-uniform: so is a column next to a zero-ghost face
    unsigned src_cols;     // bit j: column j is the source's
    int rec_lo, rec_hi;    // first and last row of the chunk's receivers in this strip (none: 1, 0)
    bool dense;            // warp-uniform: more than 32 of them; otherwise one per lane:
    int ry, rc, rid;       // its row (-1: none), column in the strip and receiver index
    float2 fx;             // sponge factors by x alone (0 outside a zero-ghost grid)
    uint32_t ring, med;    // shared-memory addresses: the warp's row slots, the lane's medium ring
    const float *tab;      // medium table
};

// column j = 0, 1 of a lane in the grid (periodic: wrapped)
__device__ __forceinline__ int col_of(const Lane &T, const StepArgs &a, int j) {
    return T.per ? wrap1(T.gx + j, a.nx) : T.gx + j;
}

// where a lane's part of population i, and of the medium, lies in a row slot
template <int Q, typename ST> __device__ __forceinline__ uint32_t slot_at(const Lane &T, int slot) {
    return T.ring + slot * slot_bytes<Q, ST>() + T.lane * 2 * (int)sizeof(ST);
}
template <int Q, typename ST> __device__ __forceinline__ uint32_t slot_med(const Lane &T, int slot) {
    return T.ring + slot * slot_bytes<Q, ST>() + Q * kCols * (int)sizeof(ST) + T.lane * 8;
}

// Copy row r into a slot: outside a zero-ghost grid zeros, across a periodic seam column by
// column.  The index bytes of an indexed medium come as the aligned word that holds them.
template <int Q, typename ST>
__device__ __forceinline__ void issue_row(const StepArgs &a, const Lane &T, int r, int slot) {
    int yw = r;
    bool live = T.live;
    if (T.per)
        yw = wrap1(r, a.ny);
    else if (r < 0 || r >= a.ny)
        live = false, yw = 0;
    const ST *in = static_cast<const ST *>(a.in);
    const uint32_t dst = slot_at<Q, ST>(T, slot), med = slot_med<Q, ST>(T, slot);
    const long long o = (long long)yw * a.pitch;
    if (!T.split) {
        const int x = live ? T.gxw : 0;
        const long long p = o + x;
#pragma unroll
        for (int i = 0; i < Q; i++)
            cp_async<2 * (int)sizeof(ST)>(dst + i * kCols * (int)sizeof(ST), in + i * a.plane + p, live);
        if (a.mid)
            cp_async<4>(med, a.mid + o + (x & ~3), live);
        else
            cp_async<8>(med, a.eta2 + p, live);
        return;
    }
    // rolled loops: this path belongs to the strips at a periodic seam, and unrolled it would
    // crowd the instruction cache of all others
    uint32_t w = 0;
#pragma unroll 1
    for (int j = 0; j < 2; j++) {
        const long long p = o + wrap1(T.gx + j, a.nx);
#pragma unroll 1
        for (int i = 0; i < Q; i++) {
            const uint32_t d = dst + (i * kCols + j) * (int)sizeof(ST);
            if constexpr (sizeof(ST) == 4) {
                cp_async<4>(d, in + i * a.plane + p, true);
            } else {
                const unsigned short v =
                    *reinterpret_cast<const unsigned short *>(in + i * a.plane + p);
                asm volatile("st.shared.u16 [%0], %1;" ::"r"(d), "h"(v) : "memory");
            }
        }
        if (a.mid)
            w |= (uint32_t)a.mid[p] << (8 * j);
        else
            cp_async<4>(med + 4 * j, a.eta2 + p, true);
    }
    // (placed as the aligned word of an unsplit lane would hold the two bytes)
    if (a.mid)
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(med), "r"(w << (8 * (T.gxw & 2))) : "memory");
}

// rho of two columns, times a level's sign
template <int Q> __device__ __forceinline__ float2 density(const float2 (&g)[Q], float sgn) {
    float2 rho = g[0];
#pragma unroll
    for (int i = 1; i < Q; i++) rho = add(rho, g[i]);
    return mul(f2(sgn), rho);
}

// first entry e of [lo, hi), ascending in rec_x, with rec_x[e] >= x: 32 samples at a time
__device__ __forceinline__ int lower_entry(const int *rec_x, int lo, int hi, int x, int lane) {
    while (lo < hi) {
        const int step = (hi - lo + 31) / 32, e = lo + lane * step;
        const int c = __popc(__ballot_sync(0xffffffffu, e < hi && rec_x[e] < x));  // samples below x
        if (step == 1 || c == 0) return lo + c;
        hi = min(hi, lo + c * step);
        lo += (c - 1) * step + 1;
    }
    return lo;
}

// The receivers of the chunk in this strip, one per lane where they are at most 32, so that the
// sweep needs no look at the lists.  scratch: 32 x 12 bytes of the warp's shared memory.
__device__ __forceinline__ void find_receivers(const WaveArgs &w, Lane &T, uint32_t scratch) {
    T.rec_lo = 1;
    T.rec_hi = 0;
    T.dense = false;
    T.ry = -1;
    if (w.row_off == nullptr) return;
    int e0 = w.row_off[T.Y0], e1 = w.row_off[T.Y1];
    if (e0 == e1) return;  // warp-uniform
    const int x0 = T.gx - 2 * T.lane;  // the strip's first column
    T.rec_lo = w.rec_y[e0];
    T.rec_hi = w.rec_y[e1 - 1];
    if (e1 - e0 > 128) {
        if (T.rec_lo != T.rec_hi) {
            T.dense = true;
            return;
        }
        e0 = lower_entry(w.rec_x, e0, e1, x0 + T.own0, T.lane);
        e1 = lower_entry(w.rec_x, e0, e1, x0 + T.own1, T.lane);
    }
    int n = 0;
    for (int e = e0 + T.lane; e - T.lane < e1; e += 32) {
        const int c = e < e1 ? w.rec_x[e] - x0 : -1;
        const bool in = c >= T.own0 && c < T.own1;
        const unsigned mask = __ballot_sync(0xffffffffu, in);
        const int k = n + __popc(mask & ((1u << T.lane) - 1u));
        if (in && k < 32)
            asm volatile("st.shared.u32 [%0], %1;\n\tst.shared.u32 [%0 + 128], %2;\n\t"
                         "st.shared.u32 [%0 + 256], %3;" ::"r"(scratch + 4 * k), "r"(w.rec_y[e]),
                         "r"(c), "r"(w.rec_id[e])
                         : "memory");
        n += __popc(mask);
    }
    if (n > 32) {
        T.dense = true;
        return;
    }
    __syncwarp();
    if (T.lane < n) {
        T.ry = (int)lds1(scratch + 4 * T.lane);
        T.rc = (int)lds1(scratch + 4 * T.lane + 128);
        T.rid = (int)lds1(scratch + 4 * T.lane + 256);
    }
    __syncwarp();
    if (n == 0) {
        T.rec_lo = 1;
        T.rec_hi = 0;
    }
}

// The receivers of row y in this strip: trace entries of time t + l.  The row's pressures go
// through one row of shared memory (`row`, 8 B a lane).
template <int Q>
__device__ __forceinline__ void record(const StepArgs &a, const WaveArgs &w, const Lane &T,
                                       const float2 (&g)[Q], float2 m, int y, int l, float sgn,
                                       uint32_t row) {
    if (!T.dense && !__any_sync(0xffffffffu, T.ry == y)) return;
    const float2 rho = density(g, sgn);
    const float px = cs2_of<Q>(e2_of<Q>(m.x), a) * rho.x, py = cs2_of<Q>(e2_of<Q>(m.y), a) * rho.y;
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(row + T.lane * 8), "f"(px), "f"(py)
                 : "memory");
    __syncwarp();
    float *out = a.trace_row + (long long)l * a.nrec;
    if (!T.dense) {
        if (T.ry == y) out[a.rec_col ? a.rec_col[T.rid] : T.rid] = __uint_as_float(lds1(row + 4 * T.rc));
    } else {
        const int x0 = T.gx - 2 * T.lane, e1 = w.row_off[y + 1];
#pragma unroll 1
        for (int e = w.row_off[y] + T.lane; e < e1; e += 32) {
            const int c = w.rec_x[e] - x0, q = w.rec_id[e];
            if (c >= T.own0 && c < T.own1)
                out[a.rec_col ? a.rec_col[q] : q] = __uint_as_float(lds1(row + 4 * c));
        }
    }
    __syncwarp();
}

// the source at row y, after the collision of level l + 1 (whose values carry sgn)
template <int Q>
__device__ __forceinline__ void add_source(const StepArgs &a, const Lane &T, float2 (&g)[Q],
                                           float2 m, int y, int l, float sgn) {
    const int yw = T.per ? wrap1(y, a.ny) : y;
    if (yw != a.src_y || a.t + l >= a.src_nt) return;  // warp-uniform
    const float S = sgn * a.src_tab[a.t + l];
    const float Sx = T.src_cols & 1u ? S : 0.f, Sy = T.src_cols & 2u ? S : 0.f;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        g[i].x += weight_i<Q>(i, e2_of<Q>(m.x), a) * Sx;
        g[i].y += weight_i<Q>(i, e2_of<Q>(m.y), a) * Sy;
    }
}

// The levels' state: what level l + 1 pulls from level l that is older than this iteration.
template <int Q, int K> struct Levels {
    static constexpr int NZ = 3, NP = Q == 5 ? 1 : 3;
    float2 z[K][NZ];     // c_y = 0 populations of level l's newest row (0, 1, 3)
    float2 p[2][K][NP];  // c_y = +1 populations (2; 2, 5, 6), by the parity of the iteration
};

// Where a lane's columns of the next rows lie: row r + kRing - 1 of the input and the medium,
// row r - K of the output (meaningful only where such a row exists).
template <typename ST> struct Rows {
    const ST *in;
    const unsigned char *mid;
    const float *eta2;
    ST *out;
};

// One wavefront iteration r of parity P.  FAST: every level's row is an output row inside the
// grid and outside the sponge, without source or receivers, the row to fetch is the next one
// in memory, and so is every lane's vector: nothing but the copies and the collisions.
// Otherwise rows [0, next_end) can be fetched so, and sp says (warp-uniform) that some row may
// hold the source or receivers.
template <int Q, int CK, int K, bool REC, typename ST, bool ROUND, bool FAST, int P>
__device__ __forceinline__ void iterate(const StepArgs &a, const WaveArgs &w, const Lane &T,
                                        Levels<Q, K> &S, Rows<ST> &at, Range<Q, ST> &range, int r,
                                        int rend, int next_end, int &slot, bool sp) {
    constexpr int NR = med_rows(K);
    cp_wait<kRing - 2>();
    float2 n[Q];  // level l's newest row r - l
    {
        const uint32_t s = slot_at<Q, ST>(T, slot);
#pragma unroll
        for (int i = 0; i < Q; i++) n[i] = range.input(i, Two<ST>::lds(s + i * kCols * (int)sizeof(ST)));
        float2 m;
        if (a.mid) {
            const uint32_t u = lds1(slot_med<Q, ST>(T, slot)) >> (8 * (T.gxw & 2));
            m = make_float2(med_of<Q>(T.tab[u & 255u]), med_of<Q>(T.tab[(u >> 8) & 255u]));
        } else {
            m = lds2(slot_med<Q, ST>(T, slot));
            m = make_float2(med_of<Q>(m.x), med_of<Q>(m.y));
        }
        const uint32_t o = T.med + (r & (NR - 1)) * kMedRow;
        if (FAST) {  // (rows in GEN iterations after this one get the factor 1 from here)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(o), "f"(m.x), "f"(m.y),
                         "f"(1.f), "f"(1.f)
                         : "memory");
        } else {
            // the factor at distance min(dx, dy) is the smaller of the two distances' factors
            int dy = min(r, a.ny - 1 - r);
            if (dy < 0 && T.per) {
                const int yw = wrap1(r, a.ny);
                dy = min(yw, a.ny - 1 - yw);
            }
            float fy = 1.f;
            if (dy < a.sponge_w) fy = dy < 0 ? 0.f : sponge_of_dist(dy, a);  // warp-uniform
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(o), "f"(m.x), "f"(m.y),
                         "f"(fminf(T.fx.x, fy)), "f"(fminf(T.fx.y, fy))
                         : "memory");
        }
    }
    // the row two ahead goes where the row before this one was read
    const int free_slot = slot == 0 ? kRing - 1 : slot - 1;
    if (FAST || (unsigned)(r + kRing - 1) < (unsigned)next_end) {
        const uint32_t d = slot_at<Q, ST>(T, free_slot);
#pragma unroll
        for (int i = 0; i < Q; i++)
            cp_async<2 * (int)sizeof(ST)>(d + i * kCols * (int)sizeof(ST), at.in + i * a.plane, T.live);
        if (a.mid)
            cp_async<4>(slot_med<Q, ST>(T, free_slot), at.mid, T.live);
        else
            cp_async<8>(slot_med<Q, ST>(T, free_slot), at.eta2, T.live);
    } else if (r + kRing - 1 < rend) {
        issue_row<Q, ST>(a, T, r + kRing - 1, free_slot);
    }
    cp_commit();
    slot = slot == kRing - 1 ? 0 : slot + 1;
    at.in += a.pitch;
    at.mid += a.pitch;
    at.eta2 += a.pitch;
    // Cuts at zero-ghost faces (cut_left), in one place ahead of the levels, which are short of
    // registers and instruction fetch (two-layer 4096^2, 200 steps: 8390 us with the cuts in each
    // level, 10530 with levels of their own for the warps at a face, 7410 here, 6690 once those warps'
    // rows count more, outer_weight, and the kernel knows its boundary; 6850 without cuts)
    if (!FAST && !T.per && (T.face || r <= K || r >= a.ny)) {  // warp-uniform
#pragma unroll
        for (int l = 0; l < K; l++) {
            cut_right(S.z[l][1], T.gx, a.nx);
            cut_left(S.z[l][2], T.gx);
            const bool row = r - l - 1 < 1 || r - l - 1 >= a.ny;  // of the rows -1 and ny - 1
#pragma unroll
            for (int i = 0; i < Levels<Q, K>::NP; i++) S.p[P][l][i] = row ? f2(0.f) : S.p[P][l][i];
            if constexpr (Q == 9) {
                cut_right(S.p[P][l][1], T.gx, a.nx);
                cut_left(S.p[P][l][2], T.gx);
            }
        }
    }
#pragma unroll
    for (int l = 0; l < K; l++) {
        const int y = r - l - 1;  // the row level l + 1 computes
        const uint32_t o = T.med + (y & (NR - 1)) * kMedRow;
        float2 m, f;
        if (FAST)
            m = lds2(o);
        else
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(m.x), "=f"(m.y), "=f"(f.x), "=f"(f.y)
                         : "r"(o));
        float2 g[Q];
        g[0] = S.z[l][0];
        g[1] = from_left(S.z[l][1]);
        g[3] = from_right(S.z[l][2]);
        g[2] = S.p[P][l][0];
        g[4] = n[4];
        S.z[l][0] = n[0];
        S.z[l][1] = n[1];
        S.z[l][2] = n[3];
        S.p[P][l][0] = n[2];
        if constexpr (Q == 9) {
            if (!FAST && !T.per) {
                cut_left(n[7], T.gx);
                cut_right(n[8], T.gx, a.nx);
            }
            g[5] = from_left(S.p[P][l][1]);
            g[6] = from_right(S.p[P][l][2]);
            g[7] = from_right(n[7]);
            g[8] = from_left(n[8]);
            S.p[P][l][1] = n[5];
            S.p[P][l][2] = n[6];
        }
        if (REC && a.rho_out && T.own && (FAST || (y >= T.Y0 && y < T.Y1)))
            Two<float>::store(a.rho_out + l * a.rho_stride + (long long)y * a.pitch + T.gx,
                              density(g, sign<CK>(l)));
        if (!FAST && sp && y >= T.rec_lo && y <= T.rec_hi)
            record<Q>(a, w, T, g, m, y, l, sign<CK>(l),  // (the next row's part of the ring is free)
                      T.med - T.lane * 16 + ((r + 1) & (NR - 1)) * kMedRow);
        collide<Q, CK>(g, m, a);
        if (!FAST) {
            if (sp && T.src) add_source<Q>(a, T, g, m, y, l, sign<CK>(l + 1));
#pragma unroll
            for (int i = 0; i < Q; i++) g[i] = mul(g[i], f);
        }
#pragma unroll
        for (int i = 0; i < Q; i++) n[i] = ROUND && l + 1 < K ? range.between(i, g[i], FAST || (y >= T.Y0 && y < T.Y1)) : g[i];
    }
    // level K holds row r - K: an output row from Y0 on
    static_assert(CK != kLossless || K % 2 == 0, "the last level's sign");
    if (T.own && (FAST || r - K >= T.Y0)) {
        if (!FAST && T.gx + 1 >= a.nx) {  // the column beyond the last
#pragma unroll
            for (int i = 0; i < Q; i++) n[i].y = 0.f;
        }
#pragma unroll
        for (int i = 0; i < Q; i++) Two<ST>::store(at.out + i * a.plane, range.output(i, n[i]));
    }
    at.out += a.pitch;
}

// One strip and row chunk of a grid.  smem: this warp's warp_bytes(); tab: room for the CTA's
// medium table.  Every warp of the CTA calls it (one barrier); those beyond the tasks do nothing.
template <int Q, int CK, int K, bool REC, typename ST, bool ROUND, int BOUND>
__device__ __forceinline__ void sweep(const StepArgs &a, const WaveArgs &w, int task,
                                      unsigned char *smem, float *tab) {
    if (a.mid)  // 8 B a thread
        cp_async<8>((uint32_t)__cvta_generic_to_shared(tab) + 8 * threadIdx.x,
                    a.mid_tab + 2 * threadIdx.x, true);
    cp_commit();
    Lane T;
    // the tasks of the outermost strips come first, then the others, strips fastest
    int bx, by;
    const int edge = w.edge_l + w.edge_r, inner = w.strips - edge, ne = edge * w.chunks_e;
    const bool outer = task < ne;
    if (outer) {
        by = task / edge;
        bx = task - by * edge;
        if (bx >= w.edge_l) bx += inner;
    } else {
        by = inner ? (task - ne) / inner : 0;
        bx = w.edge_l + (task - ne) - by * inner;
    }
    T.lane = threadIdx.x & 31;
    T.per = BOUND == kEither ? w.per != 0 : BOUND == kPeriodic;
    T.gx = bx * out_cols(K) - halo(K) + 2 * T.lane;
    T.gxw = T.gx;
    T.live = true;
    T.split = false;
    if (T.per) {
        T.gxw = wrap1(T.gx, a.nx);
        T.split = (T.gxw & 1) != 0 || T.gxw + 1 >= a.nx;
    } else {
        T.live = T.gx >= 0 && T.gx < a.nx;
    }
    T.own = T.lane >= halo(K) / 2 && T.lane < 32 - halo(K) / 2 && T.gx < a.nx;
    T.own0 = halo(K);
    T.own1 = min(kCols - halo(K), a.nx - (bx * out_cols(K) - halo(K)));
    T.Y0 = T.Y1 = 0;
    if (task < w.tasks) {
        const int n = outer ? w.chunks_e : w.chunks;
        T.Y0 = chunk_row(by, n, a.ny, a.sponge_w, w.outer, outer);
        T.Y1 = chunk_row(by + 1, n, a.ny, a.sponge_w, w.outer, outer);
    }
    T.ring = (uint32_t)__cvta_generic_to_shared(smem);
    T.med = T.ring + kRing * slot_bytes<Q, ST>() + T.lane * 16;
    T.tab = tab;
    // Rows outside a level's valid range (the first iterations) are computed from what is not
    // there yet and never reach a valid row: row y of level l takes rows y - 1 .. y + 1 of level
    // l - 1, and valid rows of level l start at Y0 - K + l.
    const int rbeg = T.Y0 - K, rend = T.Y1 + K;
    const bool work = T.Y1 > T.Y0;
#pragma unroll 1
    for (int k = 0; k < kRing - 1; k++) {
        if (work && rbeg + k < rend) issue_row<Q, ST>(a, T, rbeg + k, k);
        cp_commit();
    }
    // while these are on their way: what the sweep needs to know of the strip
    T.src_cols = 0;
    bool xedge = false;  // a column in the sponge or outside a zero-ghost grid
    float f[2];
#pragma unroll
    for (int j = 0; j < 2; j++) {
        const int x = col_of(T, a, j), d = min(x, a.nx - 1 - x);
        xedge = xedge || d < a.sponge_w;  // sponge_w >= 0: outside counts
        f[j] = d < 0 ? 0.f : a.sponge_w > 0 ? sponge_of_dist(d, a) : 1.f;
        if (x == a.src_x) T.src_cols |= 1u << j;
    }
    T.fx = make_float2(f[0], f[1]);
    T.face = __any_sync(0xffffffffu, !T.per && (T.gx == 0 || T.gx == a.nx - 1 || T.gx == a.nx - 2));
    T.src = __any_sync(0xffffffffu, T.src_cols != 0) && a.src_tab != nullptr && a.t < a.src_nt;
    if (work) find_receivers(w, T, T.med - T.lane * 16);
    cp_wait<kRing - 1>();  // the table (its group came first)
    __syncthreads();
    if (!work) return;
    Levels<Q, K> S;
#pragma unroll
    for (int l = 0; l < K; l++) {
#pragma unroll
        for (int i = 0; i < Levels<Q, K>::NZ; i++) S.z[l][i] = f2(0.f);
#pragma unroll
        for (int i = 0; i < Levels<Q, K>::NP; i++) S.p[0][l][i] = S.p[1][l][i] = f2(0.f);
    }
    // FAST iterations: [f0, f1) without those that meet the source or receiver rows
    int f0 = max(T.Y0, max(a.sponge_w, T.per ? 0 : 1)) + K;  // (1: nothing to cut)
    // (the row that an iteration takes in counts too: its sponge factor is noted as 1)
    int f1 = min(min(T.Y1 + 1, rend - kRing + 1), min(a.ny - a.sponge_w, a.ny - kRing + 1));
    if (__any_sync(0xffffffffu, xedge || T.split || (T.own && T.gx + 1 >= a.nx))) f1 = f0;
    // rows of the source and of receivers, as iterations that compute them at some level
    const int s0 = T.src ? a.src_y + 1 : rend, q0 = T.rec_lo + 1, q1 = T.rec_hi + K + 1;
    const bool has_rec = T.rec_hi >= T.rec_lo;
    auto fast_end = [&](int r) {  // iterations r .. fast_end(r) - 1 are FAST
        if (r < f0 || r >= f1) return r;
        int e = f1;
        if (T.src) {
            if (r >= s0 && r < s0 + K) return r;
            if (r < s0) e = min(e, s0);
        }
        if (has_rec) {
            if (r >= q0 && r < q1) return r;
            if (r < q0) e = min(e, q0);
        }
        return e;
    };
    Rows<ST> at;
    {
        const long long o = (long long)(rbeg + kRing - 1) * a.pitch;
        const int x = T.live ? T.gxw : 0;
        at.in = static_cast<const ST *>(a.in) + (o + x);
        at.mid = a.mid + (o + (x & ~3));
        at.eta2 = a.eta2 + (o + x);
        at.out = static_cast<ST *>(a.out) + (long long)(rbeg - K) * a.pitch + T.gx;
    }
    const bool sp = T.src || has_rec;
    const int next_end = __any_sync(0xffffffffu, T.split) ? 0 : min(a.ny, rend);
    int slot = 0;
    Range<Q, ST> range(a);
#pragma unroll 1
    for (int r = rbeg; r < rend; r += 2) {
        const int e = fast_end(r);
#pragma unroll 1
        for (; r + 1 < e; r += 2) {
            iterate<Q, CK, K, REC, ST, ROUND, true, 0>(a, w, T, S, at, range, r, rend, next_end, slot, false);
            iterate<Q, CK, K, REC, ST, ROUND, true, 1>(a, w, T, S, at, range, r + 1, rend, next_end, slot, false);
        }
        if (r >= rend) break;
        iterate<Q, CK, K, REC, ST, ROUND, false, 0>(a, w, T, S, at, range, r, rend, next_end, slot, sp);
        if (r + 1 >= rend) break;
        iterate<Q, CK, K, REC, ST, ROUND, false, 1>(a, w, T, S, at, range, r + 1, rend, next_end, slot, sp);
    }
    range.fold(a, T.lane, T.own);
}

// resident CTAs per SM the registers are cut for
template <int Q, int K, typename ST> constexpr int min_ctas() { return Q == 9 ? (K > 2 ? (sizeof(ST) == 4 ? 2 : 3) : 3) : K > 4 ? 3 : 4; }

template <int Q, int CK, int K, bool REC, typename ST, bool ROUND, int BOUND>
__global__ void __launch_bounds__(kCtaThreads, min_ctas<Q, K, ST>())
    wave_kernel(const StepArgs a, const WaveArgs w) {
    // No early launch of dependents: the next grid's CTAs would take the slots of this grid's
    // finished ones SM by SM, and leave it unevenly spread (4096^2: 38.7 us a step against 38.1,
    // 256^2: 3.1 against 2.5).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if constexpr (sizeof(ST) == 2 && K == 2)
        if (a.redo && *a.redo == 0u) return;  // (grid-uniform; FP16 only)
    extern __shared__ __align__(16) unsigned char smem[];
    float *tab = reinterpret_cast<float *>(smem + kWarpsPerCta * warp_bytes<Q, K, ST>());
    const int wi = threadIdx.x >> 5;
    sweep<Q, CK, K, REC, ST, ROUND, BOUND>(a, w, blockIdx.x * kWarpsPerCta + wi, smem + wi * warp_bytes<Q, K, ST>(), tab);
}

template <bool MRT, int K, typename ST, bool ROUND, int BOUND>
__device__ __forceinline__ void sweep_shot(const StepArgs &a, const WaveArgs &w, int block,
                                           unsigned char *smem) {
    float *tab = reinterpret_cast<float *>(smem + kWarpsPerCta * warp_bytes<5, K, ST>());
    const int wi = threadIdx.x >> 5, task = block * kWarpsPerCta + wi;
    unsigned char *mine = smem + wi * warp_bytes<5, K, ST>();
    if constexpr (MRT) {
        sweep<5, kMrt, K, true, ST, ROUND, BOUND>(a, w, task, mine, tab);
    } else {  // (block-uniform)
        if (a.omega == 2.f)
            sweep<5, kLossless, K, true, ST, ROUND, BOUND>(a, w, task, mine, tab);
        else
            sweep<5, kBgk, K, true, ST, ROUND, BOUND>(a, w, task, mine, tab);
    }
}

// Several independent D2Q5 grids ("shots") advanced by K steps in one launch: shot k owns blocks
// [first[k], first[k + 1]) and reads its own descriptors (the served batches).  FP32 and BF16 shots
// share the launch (ROUND: the BF16 ones round at every step): a few small shots leave most of
// the chip idle, and a launch of K steps takes its 10 us
// however few they are (24 shots of 256^2 to 1024^2, 400 steps: 41 ms against 47 apart).  Shots of one
// boundary and three CTAs per SM (146 registers): one kernel for both boundaries spills 572 B at four,
// one for each 356 B (32 shots of 512^2: 274 and 266 shots/s against 357).
constexpr int kBatchCtas = 3;
template <bool MRT, int K, bool ROUND, int BOUND>
__global__ void __launch_bounds__(kCtaThreads, kBatchCtas)
    wave_batch_kernel(const StepArgs *__restrict__ args, const WaveArgs *__restrict__ waves,
                      const int *__restrict__ first, int nshots) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ StepArgs sa;
    __shared__ WaveArgs sw;
    __shared__ int s_blk;
    if (threadIdx.x == 0) {
        int lo = 0, hi = nshots - 1;  // shot with first[k] <= blockIdx.x < first[k + 1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= (int)blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        sa = args[lo];
        sw = waves[lo];
        s_blk = (int)blockIdx.x - first[lo];
    }
    __syncthreads();
    if (sw.bf16)  // (block-uniform)
        sweep_shot<MRT, K, __nv_bfloat16, ROUND, BOUND>(sa, sw, s_blk, smem);
    else
        sweep_shot<MRT, K, float, false, BOUND>(sa, sw, s_blk, smem);
}

using WaveFn = void (*)(const StepArgs, const WaveArgs);
using WaveBatchFn = void (*)(const StepArgs *, const WaveArgs *, const int *, int);

}  // namespace lbwave
