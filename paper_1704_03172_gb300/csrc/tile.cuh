// tile.cuh -- K fused steps per launch for D2Q5 on register-resident tiles.
//
// A CTA of 16 warps takes a region of 64 x 64 sites: its output tile and a halo of K sites on
// every side, recomputed.  Warp v holds rows 4 v .. 4 v + 3, two columns a lane, all five
// populations of a site in registers for all K steps: a step is the collision of four rows, two
// shuffles a row for the x neighbours, and one row up and one row down through shared memory
// at the warp's edges, with one barrier.  The medium stays in shared memory.
//
// What bounds it and why this shape: the one-step kernels take 3 us a step however small the
// grid (launch and one block's chain of loads), the row wavefront (wave.cuh) 10 us a launch and
// 2K warm-up rows per chunk.  A tile step is 0.26 us of FP32 pipe (17 operations a site at 128
// lanes) and takes about 0.54, and the loads, stores and the launch around K steps about 5.
// Its price is the halo, (64 / (64 - 2K))^2, so it suits grids up to about two tiles per SM
// best and loses to the wavefront where HBM is the limit (4096^2: 383 GLUPS against 580).
// Eight warps of eight rows measured 10 to 25 % slower on small grids.  us a step, GB300, one
// step per launch / wavefront / tiles: 128^2 periodic 3.0 / 3.5 / 0.75, 512^2 5.3 / 3.4 / 1.1,
// 1024^2 6.5 / 5.0 / 3.5, 1531 x 1187 9.7 / 6.4 / 5.3, 2048^2 27 / 10.8 / 11.0.
//
// The arithmetic of a site is that of the one-step kernels, and BF16 storage is rounded at every
// step: the results are theirs bit for bit.
#pragma once

#include "wave.cuh"

namespace lbtile {

using namespace lbwave;

constexpr int kTileWarps = 16, kRows = 4;  // warps per CTA, rows per warp
constexpr int kSide = 64;              // region side
constexpr int kTileThreads = 32 * kTileWarps;
static_assert(kSide == kTileWarps * kRows && kSide == 64, "whole rows, two columns a lane");

__host__ __device__ constexpr int halo_x(int K) { return (K + 1) / 2 * 2; }  // whole lanes

struct TileArgs {
    WaveArgs rec;  // the receivers' row lists and the periodic flag (the rest unused)
    int K;         // steps
    int tx;        // tiles per row of tiles
};

// two columns of one row, from column gx on (even)
template <typename ST> __device__ __forceinline__ float2 load2(const ST *p);
template <> __device__ __forceinline__ float2 load2<float>(const float *p) {
    return *reinterpret_cast<const float2 *>(p);
}
template <> __device__ __forceinline__ float2 load2<__nv_bfloat16>(const __nv_bfloat16 *p) {
    return Two<__nv_bfloat16>::unpack(*reinterpret_cast<const uint32_t *>(p));
}

struct Shared {
    float2 edge[2][kTileWarps][2][32];   // by parity: each warp's top row's h_2 and bottom row's h_4
    float2 med[kSide][32];            // the medium (w_1), read by the lane that wrote it
    float2 factor[kSide][32];         // GEN: sponge factors (0 outside a zero-ghost grid), likewise
    float2 row[kTileWarps][48];          // a warp's row of pressures; its receivers while listing them
};

// What a warp's rows need beyond the collision: nothing; sponge factors; the source or receivers too.
enum { kPlain = 0, kEdge = 1, kSpecial = 2 };

// One step (level l + 1) of a warp's rows, from the rows next to them: the neighbours' edges.
// Apart from kSpecial there is no branch, so the rows' chains overlap.
template <int CK, bool REC, typename ST, int WHAT>
__device__ __forceinline__ void tile_rows(const StepArgs &a, const TileArgs &w, const Lane &T,
                                          Shared &sh, float2 (&h)[kRows][5], float2 up, float2 above,
                                          int y0, int l, unsigned src_rows, unsigned rec_rows) {
    const int v = threadIdx.x >> 5;
    const float sgn = CK == kLossless && (l & 1) ? -1.f : 1.f;  // of what this step pulls
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        float2 g[5];
        g[0] = h[j][0];
        g[1] = from_left(h[j][1]);
        g[2] = up;
        g[3] = from_right(h[j][3]);
        g[4] = j + 1 < kRows ? h[j + 1 < kRows ? j + 1 : 0][4] : above;
        up = h[j][2];
        const float2 m = sh.med[v * kRows + j][T.lane];
        if (REC) {
            if (T.own && y0 + j >= T.Y0 && y0 + j < T.Y1)
                Two<float>::store(a.rho_out + l * a.rho_stride + (long long)(y0 + j) * a.pitch + T.gx,
                                  density(g, sgn));
        }
        if (WHAT == kSpecial && (rec_rows >> j & 1u))  // warp-uniform
            record<5>(a, w.rec, T, g, m, y0 + j, l, sgn,
                      (uint32_t)__cvta_generic_to_shared(&sh.row[v][0]));
        collide<5, CK>(g, m, a);
        if (WHAT == kSpecial && (src_rows >> j & 1u))
            add_source<5>(a, T, g, m, y0 + j, l, CK == kLossless ? -sgn : 1.f);
        if (WHAT != kPlain) {
            const float2 f = sh.factor[v * kRows + j][T.lane];
#pragma unroll
            for (int i = 0; i < 5; i++) g[i] = mul(g[i], f);
        }
#pragma unroll
        for (int i = 0; i < 5; i++) h[j][i] = Two<ST>::round(g[i]);
    }
}

template <int CK, bool REC, typename ST, bool PER>
__device__ __forceinline__ void tile_body(const StepArgs &a, const TileArgs &w, int tile, Shared &sh) {
    const int K = w.K, hx = halo_x(K), outx = kSide - 2 * hx, outy = kSide - 2 * K;
    const int by = tile / w.tx, bx = tile - by * w.tx, v = threadIdx.x >> 5;
    Lane T;
    T.lane = threadIdx.x & 31;
    T.per = PER;
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
    T.own0 = hx;
    T.own1 = min(kSide - hx, a.nx - x0);
    T.own = 2 * T.lane >= hx && 2 * T.lane < T.own1;
    T.Y0 = max(y0, by * outy);
    T.Y1 = max(T.Y0, min(min(y0 + kRows, by * outy + outy), a.ny));
    // the state and the medium, every load in flight at once
    float2 h[kRows][5], m[kRows];
    const ST *in = static_cast<const ST *>(a.in);
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        const int y = T.per ? wrap1(y0 + j, a.ny) : y0 + j;
        const bool ok = T.live && y >= 0 && y < a.ny;
        const long long o = (long long)y * a.pitch + T.gxw;
#pragma unroll
        for (int i = 0; i < 5; i++) h[j][i] = f2(0.f);
        m[j] = f2(0.f);
        if (ok && !T.split) {
#pragma unroll
            for (int i = 0; i < 5; i++) h[j][i] = load2(in + i * a.plane + o);
            if (a.mid)
                m[j].x = __uint_as_float(*reinterpret_cast<const unsigned short *>(a.mid + o));
            else
                m[j] = load2(a.eta2 + o);
        }
    }
    if (T.split) {  // the lanes at a periodic seam, column by column
#pragma unroll
        for (int j = 0; j < kRows; j++) {
            const long long r = (long long)wrap1(y0 + j, a.ny) * a.pitch;
            const int xa = T.gxw, xb = wrap1(T.gx + 1, a.nx);
#pragma unroll
            for (int i = 0; i < 5; i++)
                h[j][i] = make_float2(Store<ST>::load1(in + i * a.plane + r + xa),
                                      Store<ST>::load1(in + i * a.plane + r + xb));
            if (a.mid)
                m[j].x = __uint_as_float((unsigned)a.mid[r + xa] | (unsigned)a.mid[r + xb] << 8);
            else
                m[j] = make_float2(a.eta2[r + xa], a.eta2[r + xb]);
        }
    }
    // whether the region meets the sponge or a zero-ghost face, the source or receivers
    const int ylo = by * outy - K, sw = a.sponge_w;
    const bool faces = !T.per || sw > 0;
    const bool gen = faces && (x0 < sw || x0 + kSide > a.nx - sw || ylo < sw || ylo + kSide > a.ny - sw);
    unsigned src_rows = 0, rec_rows = 0;
    T.src_cols = 0;
    if (a.src_tab != nullptr && a.t < a.src_nt) {
#pragma unroll
        for (int j = 0; j < 2; j++)
            if (col_of(T, a, j) == a.src_x) T.src_cols |= 1u << j;
        if (__any_sync(0xffffffffu, T.src_cols != 0)) {
#pragma unroll
            for (int j = 0; j < kRows; j++)
                if ((T.per ? wrap1(y0 + j, a.ny) : y0 + j) == a.src_y) src_rows |= 1u << j;
        }
    }
    T.src = src_rows != 0;
    T.rec_lo = 1;
    T.rec_hi = 0;
    if (T.Y1 > T.Y0) find_receivers(w.rec, T, (uint32_t)__cvta_generic_to_shared(&sh.row[v][0]));
    if (T.rec_hi >= T.rec_lo) {
#pragma unroll
        for (int j = 0; j < kRows; j++)
            if (y0 + j >= T.rec_lo && y0 + j <= T.rec_hi) rec_rows |= 1u << j;
    }
    const bool special = (src_rows | rec_rows) != 0;  // warp-uniform
    if (gen || special) {
#pragma unroll
        for (int j = 0; j < kRows; j++) {
            const int y = T.per ? wrap1(y0 + j, a.ny) : y0 + j, dy = min(y, a.ny - 1 - y);
            float f[2];
#pragma unroll
            for (int c = 0; c < 2; c++) {
                const int x = col_of(T, a, c), d = min(min(x, a.nx - 1 - x), dy);
                f[c] = d < 0 ? 0.f : sw > 0 ? sponge_of_dist(d, a) : 1.f;
            }
            sh.factor[v * kRows + j][T.lane] = make_float2(f[0], f[1]);  // (read by this lane only)
        }
    }
#pragma unroll
    for (int j = 0; j < kRows; j++) {
        if (a.mid) {
            const unsigned u = __float_as_uint(m[j].x);
            m[j] = make_float2(a.mid_tab[u & 255u], a.mid_tab[u >> 8]);
        }
        sh.med[v * kRows + j][T.lane] = make_float2(med_of<5>(m[j].x), med_of<5>(m[j].y));
    }
    // zero-ghost faces among the warp's columns and rows: cut (wave.cuh: cut_left)
    const bool left = !T.per && x0 <= 0, right = !T.per && x0 + kSide >= a.nx - 1,
               rows = !T.per && ((y0 <= 0 && y0 + kRows > 0) || (y0 < a.ny && y0 + kRows >= a.ny));
#pragma unroll 1
    for (int l = 0; l < K; l++) {
        const int par = l & 1;
        if (left) {  // warp-uniform, as the next two
#pragma unroll
            for (int j = 0; j < kRows; j++) cut_left(h[j][3], T.gx);
        }
        if (right) {
#pragma unroll
            for (int j = 0; j < kRows; j++) cut_right(h[j][1], T.gx, a.nx);
        }
        if (rows) {
#pragma unroll
            for (int j = 0; j < kRows; j++) {
                h[j][2] = y0 + j == a.ny - 1 ? f2(0.f) : h[j][2];
                h[j][4] = y0 + j == 0 ? f2(0.f) : h[j][4];
            }
        }
        sh.edge[par][v][0][T.lane] = h[kRows - 1][2];
        sh.edge[par][v][1][T.lane] = h[0][4];
        __syncthreads();  // (by parity: the next step's edges overwrite those of the step before)
        // beyond the region: part of the halo that is not used any more
        const float2 up = v > 0 ? sh.edge[par][v - 1][0][T.lane] : f2(0.f);
        const float2 above = v + 1 < kTileWarps ? sh.edge[par][v + 1][1][T.lane] : f2(0.f);
        if (special)  // warp-uniform
            tile_rows<CK, REC, ST, kSpecial>(a, w, T, sh, h, up, above, y0, l, src_rows, rec_rows);
        else if (gen)
            tile_rows<CK, REC, ST, kEdge>(a, w, T, sh, h, up, above, y0, l, 0u, 0u);
        else
            tile_rows<CK, REC, ST, kPlain>(a, w, T, sh, h, up, above, y0, l, 0u, 0u);
    }
    const float sgn = CK == kLossless && (K & 1) ? -1.f : 1.f;
    if (T.own) {
        ST *out = static_cast<ST *>(a.out);
        const bool pad = T.gx + 1 >= a.nx;  // the column beyond the last
#pragma unroll
        for (int j = 0; j < kRows; j++)
            if (y0 + j >= T.Y0 && y0 + j < T.Y1) {
#pragma unroll
                for (int i = 0; i < 5; i++) {
                    float2 q = mul(h[j][i], f2(sgn));
                    if (pad) q.y = 0.f;
                    Two<ST>::store(out + i * a.plane + (long long)(y0 + j) * a.pitch + T.gx, q);
                }
            }
    }
}

// CTAS: 1 (112 registers) where the tiles are no more than the SMs, else 2 per SM (64 registers,
// with spills, and still faster: 1024^2 3.5 against 3.7 us a step, 2048^2 11.0 against 14.9)
template <int CK, bool REC, typename ST, int CTAS, bool PER>
__global__ void __launch_bounds__(kTileThreads, CTAS) tile_kernel(const StepArgs a, const TileArgs w) {
    extern __shared__ __align__(16) unsigned char smem[];
    Shared &sh = *reinterpret_cast<Shared *>(smem);
    asm volatile("griddepcontrol.wait;" ::: "memory");  // (no early launch of dependents: wave.cuh)
    tile_body<CK, REC, ST, PER>(a, w, blockIdx.x, sh);
}

using TileFn = void (*)(const StepArgs, const TileArgs);

template <typename ST, int CTAS, bool PER> TileFn pick_tile_c(int ck, bool rec) {
    if (ck == kMrt)
        return rec ? tile_kernel<kMrt, true, ST, CTAS, PER> : tile_kernel<kMrt, false, ST, CTAS, PER>;
    if (ck == kLossless)
        return rec ? tile_kernel<kLossless, true, ST, CTAS, PER>
                   : tile_kernel<kLossless, false, ST, CTAS, PER>;
    return rec ? tile_kernel<kBgk, true, ST, CTAS, PER> : tile_kernel<kBgk, false, ST, CTAS, PER>;
}
template <typename ST> TileFn pick_tile(int ck, bool rec, int ctas, bool per) {
    if (per) return ctas == 1 ? pick_tile_c<ST, 1, true>(ck, rec) : pick_tile_c<ST, 2, true>(ck, rec);
    return ctas == 1 ? pick_tile_c<ST, 1, false>(ck, rec) : pick_tile_c<ST, 2, false>(ck, rec);
}
TileFn pick_tile_f32(int ck, bool rec, int ctas, bool per);   // tile.cu
TileFn pick_tile_bf16(int ck, bool rec, int ctas, bool per);  // tile_bf16.cu

}  // namespace lbtile
