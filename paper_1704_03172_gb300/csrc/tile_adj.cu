// tile_adj.cu -- K levels of the D2Q5 adjoint per launch on register-resident tiles.
//
// One adjoint level pulls a_j(x) = a_j(x - c_j), a_j = lambda_{opp(j)}, as a forward step pulls its
// populations (adjoint5.cu), so the tiles of tile.cuh carry over: a CTA of 16 warps holds the a_j
// of 64 x 64 sites, halo of K included, in registers for K <= 8 levels; x neighbours come by
// shuffle, rows beyond the warp's four through shared memory, one barrier a level.  rho of the
// next level comes by cp.async while this one is computed.  The medium gradient's terms are
// summed in FP32 over four levels at a time, as the wavefront sums them, and in FP64 from there.
// The levels that are left over where four do not divide a sweep are multiplied and summed in
// FP64 (WIDE), as the one-level kernel (adjoint.cu) does: a sum of few terms may cancel.
//
// What bounds it and why this shape: issue, and the barrier.  A wavefront launch takes its rows one
// after another and needs 2 K of them to start with, which small grids cannot hide.  1201 x 911
// (7 levels a launch, two CTAs per SM): 9.6 us a level against 11; 2048^2: 27.4 against 23.4, so
// the line is drawn at the forward tiles' 3.5 million sites.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "adjoint_site.cuh"
#include "lb_kernels.cuh"
#include "lb_runtime.h"
#include "tile.cuh"

namespace lbtileadj {

using namespace lbk;
using namespace lbadj;
using namespace lbtile;

constexpr int kLevels = 8;  // at most: two FP32 sums of four levels

struct TileAdjArgs {
    const float *rho_hi;  // rho(x, t_hi); level l (from 0) reads rho_hi - l plane
    long long t_hi;       // time of level 0
    WaveArgs rec;         // the receivers' row lists and the periodic flag (the rest unused)
    int K, tx;
};

struct SharedAdj {
    float2 edge[2][kTileWarps][2][32];  // by parity: each warp's last row's a_2 and first row's a_4
    float2 e2[kSide][32];               // eta^2; from here on read by the lane that wrote it
    float2 factor[kSide][32];           // sponge factors (0 outside a zero-ghost grid)
    float2 rho[kSide][32];              // rho of the next level (own sites; else 0)
    union {
        float2 sum[2][kSide][32];       // gradient terms of levels 0 .. 3 and 4 .. 7
        double2 wide[kSide][32];        // WIDE: of all levels
    };
    int2 rec[kSide][32];                // by column: receiver id, -1 none, -2 several
};

// adj_site for two columns
template <bool MRT>
__device__ __forceinline__ float2 site(float2 (&m)[5], float2 e2, const StepArgs &a) {
    const float2 w0 = fma(-1.f, e2, f2(1.f)), w1 = mul(f2(0.25f), e2);
    const float2 s14 = add(add(add(m[1], m[2]), m[3]), m[4]);
    if constexpr (!MRT) {
        const float om = a.omega, hb = 0.5f * om, keep = 1.f - om;
        const float2 A = mul(f2(om), fma2(w0, m[0], mul(w1, s14)));
        const float2 dx = sub(m[1], m[3]), dy = sub(m[2], m[4]);
        const float2 gsum = mul(f2(om), fma(0.25f, s14, mul(f2(-1.f), m[0])));
        m[0] = fma(keep, m[0], A);
        m[1] = fma(keep, m[1], fma(hb, dx, A));
        m[2] = fma(keep, m[2], fma(hb, dy, A));
        m[3] = fma(keep, m[3], fma(-hb, dx, A));
        m[4] = fma(keep, m[4], fma(-hb, dy, A));
        return gsum;
    } else {
        const float2 me = mul(f2(a.s[3]), fma(-4.f, m[0], s14));
        const float2 mp = mul(f2(a.s[4]), sub(add(sub(m[1], m[2]), m[3]), m[4]));
        const float2 A = mul(mul(f2(4.f), me), sub(w1, w0));
        const float2 d13 = sub(A, add(me, mp)), d24 = sub(A, sub(me, mp));
        m[0] = add(fma(4.f, me, m[0]), A);
        m[1] = add(m[1], d13);
        m[2] = add(m[2], d24);
        m[3] = add(m[3], d13);
        m[4] = add(m[4], d24);
        return mul(f2(5.f), me);
    }
}

// first of the receivers of row y with rec_x >= x
__device__ __forceinline__ int first_of(const WaveArgs &w, int y, int x) {
    int lo = w.row_off[y], hi = w.row_off[y + 1];
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (w.rec_x[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}
// the receiver at column x of row y: its id, -1 none, -2 several
__device__ __forceinline__ int receiver_at(const WaveArgs &w, int y, int x) {
    const int e = first_of(w, y, x), hi = w.row_off[y + 1];
    if (e >= hi || w.rec_x[e] != x) return -1;
    return e + 1 < hi && w.rec_x[e + 1] == x ? -2 : w.rec_id[e];
}
// the sum of dJ/dp over a site's receivers at row `row` of dJ/dp
template <typename R>
__device__ __forceinline__ R residual(const AdjArgs &d, const WaveArgs &w, int id, int y, int x,
                                      long long row) {
    if (id == -1) return 0;
    const float *p = d.resid + row * d.nrec;
    if (id >= 0) return p[id];
    R sum = 0;
    const int hi = w.row_off[y + 1];
    for (int e = first_of(w, y, x); e < hi && w.rec_x[e] == x; e++) sum += p[w.rec_id[e]];
    return sum;
}

template <bool MRT, int WHAT, bool WIDE>
__device__ __forceinline__ void level(const StepArgs &a, const AdjArgs &d, const TileAdjArgs &w,
                                      const Lane &T, SharedAdj &sh, float2 (&h)[kRows][5], float2 up,
                                      float2 above, int y0, int l, unsigned own_rows,
                                      unsigned src_rows, unsigned rec_rows) {
    const int v = threadIdx.x >> 5;
    const long long t = w.t_hi - l;
    using V = std::conditional_t<WIDE, double, float>;  // of a gradient term
    struct {
        V x, y;
    } R[kRows];
    if (WHAT == kSpecial) {  // on their way while the rows before are computed
#pragma unroll
        for (int j = 0; j < kRows; j++) {
            R[j].x = R[j].y = 0;
            if (rec_rows >> j & 1u) {  // warp-uniform
                const int2 id = sh.rec[v * kRows + j][T.lane];
                const int y = T.per ? wrap1(y0 + j, a.ny) : y0 + j;
                R[j].x = residual<V>(d, w.rec, id.x, y, col_of(T, a, 0), t - d.t0);
                R[j].y = residual<V>(d, w.rec, id.y, y, col_of(T, a, 1), t - d.t0);
            }
        }
    }
    cp_wait<0>();
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        const int row = v * kRows + j;
        // mu_i = a_{opp(i)}(x - c_{opp(i)})
        float2 m[5];
        m[0] = h[j][0];
        m[3] = from_left(h[j][1]);
        m[4] = up;
        m[1] = from_right(h[j][3]);
        m[2] = j + 1 < kRows ? h[j + 1 < kRows ? j + 1 : 0][4] : above;
        up = h[j][2];
        const float2 e2 = sh.e2[row][T.lane], rho = sh.rho[row][T.lane];
        float2 part = f2(0.f);
        double2 wide = make_double2(0., 0.);
        if (WIDE)
            wide = sh.wide[row][T.lane];
        else
            part = sh.sum[l >> 2][row][T.lane];
        if (WHAT != kPlain) {
            const float2 f = sh.factor[row][T.lane];
#pragma unroll
            for (int i = 0; i < 5; i++) m[i] = mul(m[i], f);
        }
        if (WHAT == kSpecial && (src_rows >> j & 1u)) {  // warp-uniform
#pragma unroll
            for (int c = 0; c < 2; c++) {
                if (!(T.src_cols >> c & 1u)) continue;
                const float mm[5] = {c ? m[0].y : m[0].x, c ? m[1].y : m[1].x, c ? m[2].y : m[2].x,
                                     c ? m[3].y : m[3].x, c ? m[4].y : m[4].x};
                float src_w, src_dw;
                adj_src<5>(mm, c ? e2.y : e2.x, a, src_w, src_dw);
                if (T.own && T.gx + c < a.nx && (own_rows >> j & 1u)) d.grad_src[t - d.t0] = (double)src_w;
                if (t < a.src_nt) {
                    if (WIDE)
                        (c ? wide.y : wide.x) += (double)a.src_tab[t] * (double)src_dw;
                    else
                        (c ? part.y : part.x) += a.src_tab[t] * src_dw;
                }
            }
        }
        const float2 gsum = site<MRT>(m, e2, a);
        if (WIDE) {
            wide.x += (double)rho.x * (double)gsum.x;
            wide.y += (double)rho.y * (double)gsum.y;
        } else {
            part = fma2(rho, gsum, part);
        }
        if (WHAT == kSpecial && (rec_rows >> j & 1u)) {
            const float2 R2 = make_float2((float)R[j].x, (float)R[j].y);
            const float2 Rc = make_float2(R2.x * cs2_of<5>(e2.x, a), R2.y * cs2_of<5>(e2.y, a));
#pragma unroll
            for (int i = 0; i < 5; i++) m[i] = add(m[i], Rc);
            if (WIDE) {
                wide.x += (double)R[j].x * (double)dcs2<5>(a) * (double)rho.x;
                wide.y += (double)R[j].y * (double)dcs2<5>(a) * (double)rho.y;
            } else {
                part = fma2(mul(R2, f2(dcs2<5>(a))), rho, part);
            }
        }
        if (WIDE)
            sh.wide[row][T.lane] = wide;
        else
            sh.sum[l >> 2][row][T.lane] = part;
        h[j][0] = m[0];
        h[j][1] = m[3];
        h[j][2] = m[4];
        h[j][3] = m[1];
        h[j][4] = m[2];
    }
}

// rho of level l for the warp's rows (own sites), into the lane's places
__device__ __forceinline__ void issue_rho(const StepArgs &a, const TileAdjArgs &w, const Lane &T,
                                          SharedAdj &sh, int y0, int l, unsigned own_rows) {
    const int v = threadIdx.x >> 5;
    const float *p = w.rho_hi - (long long)l * a.plane;
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        const bool own = T.own && (own_rows >> j & 1u);
        cp_async<8>((uint32_t)__cvta_generic_to_shared(&sh.rho[v * kRows + j][T.lane]),
                    own ? p + (long long)(y0 + j) * a.pitch + T.gx : w.rho_hi, own);
    }
    cp_commit();
}

// CTAS as in tile.cuh
template <bool MRT, int CTAS, bool WIDE>
__global__ void __launch_bounds__(kTileThreads, CTAS)
    tile_adj_kernel(const StepArgs a, const AdjArgs d, const TileAdjArgs w) {
    extern __shared__ __align__(16) unsigned char smem[];
    SharedAdj &sh = *reinterpret_cast<SharedAdj *>(smem);
    asm volatile("griddepcontrol.wait;" ::: "memory");  // (no early launch of dependents: wave.cuh)
    const int K = w.K, hx = halo_x(K), outx = kSide - 2 * hx, outy = kSide - 2 * K;
    const int by = (int)blockIdx.x / w.tx, bx = (int)blockIdx.x - by * w.tx, v = threadIdx.x >> 5;
    Lane T;
    T.lane = threadIdx.x & 31;
    T.per = w.rec.per != 0;
    const int x0 = bx * outx - hx, y0 = by * outy - K + v * kRows;  // the region's, the warp's first
    T.gx = x0 + 2 * T.lane;
    T.gxw = T.gx;
    T.live = true;
    T.split = false;
    if (T.per) {
        T.gxw = wrap1(T.gx, a.nx);
        T.split = (T.gxw & 1) != 0 || T.gxw + 1 >= a.nx;
    } else {
        T.live = T.gx >= 0 && T.gx < a.nx;
    }
    T.own1 = min(kSide - hx, a.nx - x0);
    T.own = 2 * T.lane >= hx && 2 * T.lane < T.own1;
    const int Y0 = max(y0, by * outy), Y1 = min(min(y0 + kRows, by * outy + outy), a.ny);
    unsigned own_rows = 0;
#pragma unroll
    for (int j = 0; j < kRows; j++) own_rows |= y0 + j >= Y0 && y0 + j < Y1 ? 1u << j : 0u;
    issue_rho(a, w, T, sh, y0, 0, own_rows);
    float2 h[kRows][5];
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        const int y = T.per ? wrap1(y0 + j, a.ny) : y0 + j;
        const bool ok = T.live && y >= 0 && y < a.ny;
        const long long o = (long long)y * a.pitch + T.gxw;
        float2 e = f2(0.f);
#pragma unroll
        for (int i = 0; i < 5; i++) h[j][i] = f2(0.f);
        if (ok && !T.split) {
#pragma unroll
            for (int i = 0; i < 5; i++) h[j][i] = load2(d.lam_in + Lat<5>::opp(i) * a.plane + o);
            e = load2(a.eta2 + o);
        } else if (ok) {  // the lanes at a periodic seam, column by column
            const long long r = (long long)y * a.pitch;
            const int xa = T.gxw, xb = wrap1(T.gx + 1, a.nx);
#pragma unroll
            for (int i = 0; i < 5; i++) {
                const float *p = d.lam_in + Lat<5>::opp(i) * a.plane + r;
                h[j][i] = make_float2(p[xa], p[xb]);
            }
            e = make_float2(a.eta2[r + xa], a.eta2[r + xb]);
        }
        sh.e2[v * kRows + j][T.lane] = e;
        if (WIDE) {
            sh.wide[v * kRows + j][T.lane] = make_double2(0., 0.);
        } else {
            sh.sum[0][v * kRows + j][T.lane] = f2(0.f);
            sh.sum[1][v * kRows + j][T.lane] = f2(0.f);
        }
    }
    // whether the region meets the sponge or a zero-ghost face, the source or receivers
    const int ylo = by * outy - K, sw = a.sponge_w;
    const bool faces = !T.per || sw > 0;
    const bool gen = faces && (x0 < sw || x0 + kSide > a.nx - sw || ylo < sw || ylo + kSide > a.ny - sw);
    unsigned src_rows = 0, rec_rows = 0;
    T.src_cols = 0;
    if (a.src_tab != nullptr) {
#pragma unroll
        for (int c = 0; c < 2; c++)
            if (col_of(T, a, c) == a.src_x) T.src_cols |= 1u << c;
    }
    const bool src = __any_sync(0xffffffffu, T.src_cols != 0);
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        const int y = T.per ? wrap1(y0 + j, a.ny) : y0 + j, dy = min(y, a.ny - 1 - y);
        float f[2];
        int id[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int x = col_of(T, a, c), dist = min(min(x, a.nx - 1 - x), dy);
            f[c] = dist < 0 ? 0.f : sw > 0 ? sponge_of_dist(dist, a) : 1.f;
            id[c] = -1;
            if (w.rec.row_off && dist >= 0 && w.rec.row_off[y + 1] > w.rec.row_off[y])
                id[c] = receiver_at(w.rec, y, x);
        }
        sh.factor[v * kRows + j][T.lane] = make_float2(f[0], f[1]);
        sh.rec[v * kRows + j][T.lane] = make_int2(id[0], id[1]);
        if (__any_sync(0xffffffffu, id[0] != -1 || id[1] != -1)) rec_rows |= 1u << j;
        if (src && y == a.src_y) src_rows |= 1u << j;
    }
    const bool special = (src_rows | rec_rows) != 0;  // warp-uniform
#pragma unroll 1
    for (int l = 0; l < K; l++) {
        const int par = l & 1;
        sh.edge[par][v][0][T.lane] = h[kRows - 1][2];
        sh.edge[par][v][1][T.lane] = h[0][4];
        __syncthreads();  // (by parity: the next level's edges overwrite those of the one before)
        // beyond the region: part of the halo that is not used any more
        const float2 up = v > 0 ? sh.edge[par][v > 0 ? v - 1 : 0][0][T.lane] : f2(0.f);
        const float2 above = v + 1 < kTileWarps ? sh.edge[par][v + 1 < kTileWarps ? v + 1 : v][1][T.lane]
                                                : f2(0.f);
        if (special)  // warp-uniform
            level<MRT, kSpecial, WIDE>(a, d, w, T, sh, h, up, above, y0, l, own_rows, src_rows, rec_rows);
        else if (gen)
            level<MRT, kEdge, WIDE>(a, d, w, T, sh, h, up, above, y0, l, own_rows, 0u, 0u);
        else
            level<MRT, kPlain, WIDE>(a, d, w, T, sh, h, up, above, y0, l, own_rows, 0u, 0u);
        if (l + 1 < K) issue_rho(a, w, T, sh, y0, l + 1, own_rows);
    }
    if (T.own) {
        const bool pad = T.gx + 1 >= a.nx;  // the column beyond the last
#pragma unroll
        for (int j = 0; j < kRows; j++) {
            if (!(own_rows >> j & 1u)) continue;
            const long long o = (long long)(y0 + j) * a.pitch + T.gx;
#pragma unroll
            for (int i = 0; i < 5; i++) {
                if (pad) h[j][i].y = 0.f;
                Two<float>::store(d.lam_out + Lat<5>::opp(i) * a.plane + o, h[j][i]);
            }
            double2 s;
            if (WIDE) {
                s = sh.wide[v * kRows + j][T.lane];
            } else {
                const float2 s0 = sh.sum[0][v * kRows + j][T.lane], s1 = sh.sum[1][v * kRows + j][T.lane];
                s = make_double2((double)s0.x + (double)s1.x, (double)s0.y + (double)s1.y);
            }
            double2 g = *reinterpret_cast<const double2 *>(d.grad + o);
            g.x += s.x;
            if (!pad) g.y += s.y;
            *reinterpret_cast<double2 *>(d.grad + o) = g;
        }
    }
}

}  // namespace lbtileadj

using namespace lbtileadj;
using namespace lbrt;

// Levels of the next launch of n wanted ones (0: the wavefront's): 4 or 8, as costs less a level
// (a tile's cost as in wave.cu's tile_cost), and what is left of four in FP64.
int tile_adj_levels(const lb_ctx *ctx, int n) {
    if ((long long)ctx->ny * ctx->pitch >= 3500000) return 0;
    if (n < 4) return n;
    auto cost = [&](int K) {
        const int ox = kSide - 2 * halo_x(K), oy = kSide - 2 * K;
        const long long t = (long long)((ctx->nx + ox - 1) / ox) * ((ctx->ny + oy - 1) / oy);
        return t <= sm_count() ? 520 + 54 * K
                               : std::max<long long>(600 + 135 * K, 400 + t * (250 + 62 * K) / sm_count());
    };
    return n >= kLevels && cost(kLevels) <= 2 * cost(4) ? kLevels : 4;
}

cudaError_t tile_adj_launch(lb_ctx *ctx, const StepArgs &a, const AdjArgs &d, const float *rho_hi,
                            long long t_hi, int K) {
    TileAdjArgs w;
    w.rho_hi = rho_hi;
    w.t_hi = t_hi;
    w.rec = WaveArgs{};
    w.rec.row_off = ctx->nrec > 0 ? ctx->row_off : nullptr;
    w.rec.rec_x = ctx->row_x;
    w.rec.rec_id = ctx->row_id;
    w.K = K;
    w.rec.per = ctx->cfg.boundary == LB_PERIODIC ? 1 : 0;
    const int ox = kSide - 2 * halo_x(K), oy = kSide - 2 * K;
    w.tx = (ctx->nx + ox - 1) / ox;
    const int tiles = w.tx * ((ctx->ny + oy - 1) / oy);
    const bool mrt = ctx->cfg.collision == LB_MRT, one = tiles <= sm_count();
    void (*fn)(const StepArgs, const AdjArgs, const TileAdjArgs);
    if (K < 4)
        fn = mrt ? (one ? tile_adj_kernel<true, 1, true> : tile_adj_kernel<true, 2, true>)
                 : (one ? tile_adj_kernel<false, 1, true> : tile_adj_kernel<false, 2, true>);
    else
        fn = mrt ? (one ? tile_adj_kernel<true, 1, false> : tile_adj_kernel<true, 2, false>)
                 : (one ? tile_adj_kernel<false, 1, false> : tile_adj_kernel<false, 2, false>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SharedAdj));
    if (e != cudaSuccess) return e;
    return launch_pdl(fn, dim3(tiles), dim3(kTileThreads), sizeof(SharedAdj), ctx->stream, a, d, w);
}
