// sweep3.cuh -- two fused D3Q7 steps per launch: a tile of columns swept along z.
//
// A CTA of 16 warps owns up to 60 x 30 sites of every plane of a chunk of planes and computes on a
// region of 64 x 32: warp v has rows 2 v and 2 v + 1, a lane two columns.  In iteration z
//   level 1  pulls plane z from h^{t-1} in memory and collides it,
//   level 2  pulls plane z - 1 from level 1 and stores it,
// so what level 2 needs of level 1 is in the lane's registers (planes z - 1 and, for c_z = +1,
// z - 2; c_z = -1 comes from the plane just computed), next to it by shuffle (x) or, at a warp's
// first and last row, in shared memory (y).  One barrier a plane.
//
// What bounds it and why this shape: the one-step kernel is bound by HBM (57 B a site and step,
// with an indexed medium); two steps in one sweep move half (ncu: 975 MB a launch at 256^3).  Rows
// come by cp.async into the lane's own place in shared memory, refilled as soon as it has been
// read, so a CTA has a whole plane (57 KB in FP32) on its way while it computes the one before.
// The pulls along y and z are made by address, those along x by shuffle; the recomputed ring (one
// site of level 1) costs at most 7 % of the arithmetic, and its loads meet the neighbouring tile's
// in L2.  What is left is the latency of a row's chain of operations, hence many warps: 16 of two
// rows at 64 registers, two CTAs per SM, took 7830 us for 60 steps at 256^3, 8 warps of four rows
// 8070 (two rows at a time, with spills: 8520), one CTA of 64 x 64 sites per SM 7925, one step per
// launch 10130; 320^3: 212 us a step against 309, BF16 162 against 290.
//
// The arithmetic of a site is that of the one-step kernels, operation by operation, and BF16
// storage is rounded at every step: the results are theirs bit for bit.
#pragma once

#include "wave.cuh"

namespace lbsweep3 {

using namespace lbwave;

constexpr int kWarpsZ = 16, kRowsZ = 2, kTake = 1;   // warps per CTA, rows per warp, rows at a time
constexpr int kRegX = 64, kRegY = kWarpsZ * kRowsZ;  // region
constexpr int kHaloX = 2, kHaloY = 1;                // x: a whole lane
constexpr int kMaxX = kRegX - 2 * kHaloX, kMaxY = kRegY - 2 * kHaloY;
constexpr int kThreadsZ = 32 * kWarpsZ;

struct SweepArgs {
    int tx, ty;      // tiles along x and y
    int outx, outy;  // their sites (outx even)
    int chunks;      // of planes
    int per;         // periodic boundary
    int rec_blocks;  // the first blocks: receivers
};

template <typename ST> struct SharedZ {
    ST pop[kRegY][7][kRegX];  // what a lane pulls next; read by the lane that copied it, as the
    float2 med[kRegY][32];    // medium: eta^2, or the index word
    float2 e2[kRegY][32];     // eta^2 of the plane before
    float2 factor[kRegY][32]; // sponge factor by x and y; -1 outside a zero-ghost grid
    float2 edge[2][kWarpsZ][2][32];  // by parity of z: each warp's last row's h_2, first row's h_4
    float tab[256];
};

// in place: g becomes h (collide7, with the fused operations it compiles to)
__device__ __forceinline__ void collide7p(float2 (&g)[7], float2 e2, float om) {
    const float2 rho = add(add(add(add(add(add(g[0], g[1]), g[2]), g[3]), g[4]), g[5]), g[6]);
    const float2 jx = sub(g[1], g[3]), jy = sub(g[2], g[4]), jz = sub(g[5], g[6]);
    const float2 b = mul(mul(e2, f2(1.f / 6.f)), rho), eq0 = fma(-6.f, b, rho);
    auto relax = [om](float2 eq, float2 h) { return fma(om, sub(eq, h), h); };
    g[0] = relax(eq0, g[0]);
    g[1] = relax(fma(0.5f, jx, b), g[1]);
    g[2] = relax(fma(0.5f, jy, b), g[2]);
    g[3] = relax(fma(-0.5f, jx, b), g[3]);
    g[4] = relax(fma(-0.5f, jy, b), g[4]);
    g[5] = relax(fma(0.5f, jz, b), g[5]);
    g[6] = relax(fma(-0.5f, jz, b), g[6]);
}

// First value of row y of plane z.  64 bits throughout: a plane alone may hold more than 2^31 sites.
__host__ __device__ constexpr long long row_start(int y, int z, int ny3, int pitch) {
    return ((long long)z * ny3 + y) * pitch;
}

// index of a row or plane in the grid: wrapped, or -1 outside a zero-ghost grid
__device__ __forceinline__ int at_or_none(int v, int n, bool per) {
    return per ? wrap1(v, n) : (unsigned)v < (unsigned)n ? v : -1;
}

// What a lane pulls for row y of plane z into its place in row `row` of the region: the general
// form (one copy in the kernel; issue_inside where every row and plane it reads lies inside).
template <typename ST>
__device__ __forceinline__ void issue(const StepArgs &a, const Lane &T, SharedZ<ST> &sh, int row,
                                      int y, int z, bool wanted) {
    const int yc = at_or_none(y, a.ny3, T.per), ym = at_or_none(y - 1, a.ny3, T.per),
              yp = at_or_none(y + 1, a.ny3, T.per);
    const int zc = at_or_none(z, a.nz, T.per), zm = at_or_none(z - 1, a.nz, T.per),
              zp = at_or_none(z + 1, a.nz, T.per);
    // by population: its row (row 0 and no bytes where there is none)
    const bool c = wanted && yc >= 0 && zc >= 0;
    const bool ok[7] = {c, c, wanted && ym >= 0 && zc >= 0, c, wanted && yp >= 0 && zc >= 0,
                        wanted && yc >= 0 && zm >= 0, wanted && yc >= 0 && zp >= 0};
    const int ys[7] = {yc, yc, ym, yc, yp, yc, yc}, zs[7] = {zc, zc, zc, zc, zc, zm, zp};
    const ST *in = static_cast<const ST *>(a.in);
    const int x = T.live ? T.gxw : 0;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sh.pop[row][0][2 * T.lane]);
#pragma unroll
    for (int i = 0; i < 7; i++) {
        const long long o = ok[i] ? row_start(ys[i], zs[i], a.ny3, a.pitch) : 0;
        cp_async<2 * (int)sizeof(ST)>(dst + i * kRegX * (int)sizeof(ST), in + i * a.plane + o + x,
                                      ok[i] && T.live);
    }
    const long long o = c ? row_start(yc, zc, a.ny3, a.pitch) : 0;
    const uint32_t med = (uint32_t)__cvta_generic_to_shared(&sh.med[row][T.lane]);
    if (a.mid)
        cp_async<4>(med, a.mid + o + (x & ~3), c && T.live);
    else
        cp_async<8>(med, a.eta2 + o + x, c && T.live);
}

// The same where no row, plane or column wraps.
// at0: row y's first value in plane z (the same for all lanes); lane: the lane's columns in the row.
// CHECK: rows and planes may lie outside a zero-ghost grid; otherwise they all lie inside.
template <typename ST, bool CHECK>
__device__ __forceinline__ void issue_inside(const StepArgs &a, const Lane &T, SharedZ<ST> &sh, int row,
                                             int y, int z, long long at0, int lane) {
    const long long dz = row_start(0, 1, a.ny3, a.pitch);
    const long long by[7] = {0, 0, -(long long)a.pitch, 0, a.pitch, -dz, dz};
    bool c = T.live, ok[7] = {c, c, c, c, c, c, c};
    if (CHECK) {
        const bool yc = (unsigned)y < (unsigned)a.ny3, zc = (unsigned)z < (unsigned)a.nz;
        c = c && yc && zc;
        ok[0] = ok[1] = ok[3] = c;
        ok[2] = T.live && zc && (unsigned)(y - 1) < (unsigned)a.ny3;
        ok[4] = T.live && zc && (unsigned)(y + 1) < (unsigned)a.ny3;
        ok[5] = T.live && yc && (unsigned)(z - 1) < (unsigned)a.nz;
        ok[6] = T.live && yc && (unsigned)(z + 1) < (unsigned)a.nz;
    }
    const ST *in = static_cast<const ST *>(a.in);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sh.pop[row][0][2 * T.lane]);
#pragma unroll
    for (int i = 0; i < 7; i++) {
        const ST *from = in + (at0 + (i * a.plane + by[i])) + lane;
        if (CHECK && !ok[i]) from = in;
        cp_async<2 * (int)sizeof(ST)>(dst + i * kRegX * (int)sizeof(ST), from, ok[i]);
    }
    const uint32_t med = (uint32_t)__cvta_generic_to_shared(&sh.med[row][T.lane]);
    const long long m = CHECK && !c ? 0 : at0 + lane;
    if (a.mid)
        cp_async<4>(med, a.mid + (m & ~3LL), c);
    else
        cp_async<8>(med, a.eta2 + m, c);
}

// 0 outside a zero-ghost grid (f < 0), whatever was computed there: a product with 0 would keep a
// non-finite value, which the one-step kernels lose across the face
__device__ __forceinline__ float2 inside_only(float2 v, float2 f) {
    return make_float2(f.x < 0.f ? 0.f : v.x, f.y < 0.f ? 0.f : v.y);
}

// What a plane's rows need beyond the collisions: nothing, or sponge factors, zeros outside a
// zero-ghost grid and the source.
enum { kInside = 0, kEdges = 1 };

// source and sponge of a row after its collision; f: its factors, -1 outside; out: some may be
template <int WHAT>
__device__ __forceinline__ void finish(const StepArgs &a, const Lane &T, float2 (&g)[7], float2 e2,
                                       float2 f, bool out, bool src, int l) {
    if (WHAT == kInside) return;
    if (src && a.t + l < a.src_nt) {  // warp-uniform
        const float S = a.src_tab[a.t + l];
        const float Sx = T.src_cols & 1u ? S : 0.f, Sy = T.src_cols & 2u ? S : 0.f;
#pragma unroll
        for (int i = 0; i < 7; i++) {
            g[i].x += weight_i<7>(i, e2.x, a) * Sx;
            g[i].y += weight_i<7>(i, e2.y, a) * Sy;
        }
    }
#pragma unroll
    for (int i = 0; i < 7; i++) g[i] = mul(g[i], f);
    if (out) {  // CTA-uniform
#pragma unroll
        for (int i = 0; i < 7; i++) g[i] = inside_only(g[i], f);
    }
}

// factor of plane z (-1 outside a zero-ghost grid)
__device__ __forceinline__ float plane_factor(const StepArgs &a, int z, bool per) {
    const int zw = at_or_none(z, a.nz, per);
    return zw < 0 ? -1.f : a.sponge_w > 0 ? sponge_of_dist(min(zw, a.nz - 1 - zw), a) : 1.f;
}

// One plane of a warp's rows.  H: level 1's populations 0 .. 4 of plane z - 1, H5: population 5 of
// planes z - 2 and z - 1; both move on by a plane.  next: whether plane z + 1 is fetched here, row
// j's from at0 + j pitch on; out0: row 0 of plane z - 1.
template <typename ST, int WHAT>
__device__ __forceinline__ void plane(const StepArgs &a, const Lane &T, SharedZ<ST> &sh,
                                      float2 (&H)[kRowsZ][5], float2 (&H5)[2][kRowsZ], int v, int y0, int z,
                                      bool next, long long at0, int from, bool level2, long long out0, int lane,
                                      unsigned own_rows, bool out, unsigned src1, unsigned src0) {
    const int par = z & 1;
    // beyond the region: part of the halo that is not used any more
    float2 up = v > 0 ? sh.edge[par ^ 1][v > 0 ? v - 1 : 0][0][T.lane] : f2(0.f);
    const float2 above = v + 1 < kWarpsZ ? sh.edge[par ^ 1][v + 1 < kWarpsZ ? v + 1 : v][1][T.lane]
                                         : f2(0.f);
    float f1 = 1.f, f0 = 1.f;
    if (WHAT != kInside) {
        f1 = plane_factor(a, z, T.per);
        f0 = plane_factor(a, z - 1, T.per);
    }
    const float om = a.omega;
#pragma unroll
    for (int j0 = 0; j0 < kRowsZ; j0 += kTake) {
        cp_wait<kRowsZ / kTake - 1>();
        float2 g[kTake][7], e[kTake], ep[kTake], fxy[kTake];
#pragma unroll
        for (int p = 0; p < kTake; p++) {
            const int row = v * kRowsZ + j0 + p;
            const uint32_t at = (uint32_t)__cvta_generic_to_shared(&sh.pop[row][0][2 * T.lane]);
#pragma unroll
            for (int k = 0; k < 7; k++) {
                const int i = k < 4 ? (k < 2 ? 2 * k : k == 2 ? 4 : 5) : k == 4 ? 6 : k == 5 ? 1 : 3;
                g[p][i] = Two<ST>::lds(at + i * kRegX * (int)sizeof(ST));  // 1 and 3, shuffled, last
            }
            e[p] = sh.med[row][T.lane];
            if (a.mid) {
                const unsigned u = __float_as_uint(e[p].x) >> (8 * (T.gxw & 2));
                e[p] = make_float2(sh.tab[u & 255u], sh.tab[(u >> 8) & 255u]);
            }
            ep[p] = sh.e2[row][T.lane];
            sh.e2[row][T.lane] = e[p];
            fxy[p] = WHAT != kInside ? sh.factor[row][T.lane] : f2(1.f);
        }
#pragma unroll
        for (int p = 0; p < kTake; p++) {
            g[p][1] = from_left(g[p][1]);
            g[p][3] = from_right(g[p][3]);
        }
        // (after the shuffles: the rows have been read)
        if (next) {
#pragma unroll
            for (int p = 0; p < kTake; p++)
                issue_inside<ST, WHAT != kInside>(a, T, sh, v * kRowsZ + j0 + p, y0 + j0 + p, z + 1,
                                                  at0 + (long long)(j0 + p) * a.pitch, from);
        }
        cp_commit();
#pragma unroll
        for (int p = 0; p < kTake; p++) {
            collide7p(g[p], e[p], om);
            finish<WHAT>(a, T, g[p], e[p], make_float2(fminf(fxy[p].x, f1), fminf(fxy[p].y, f1)), out,
                         src1 >> (j0 + p) & 1u, 0);
#pragma unroll
            for (int i = 0; i < 7; i++) g[p][i] = Two<ST>::round(g[p][i]);
        }
#pragma unroll
        for (int p = 0; p < kTake; p++) {
            const int j = j0 + p;
            if (level2) {  // CTA-uniform: plane z - 1 is an output plane
                float2 q[7];
                q[0] = H[j][0];
                q[1] = from_left(H[j][1]);
                q[2] = up;
                q[3] = from_right(H[j][3]);
                q[4] = j + 1 < kRowsZ ? H[j + 1 < kRowsZ ? j + 1 : 0][4] : above;
                q[5] = H5[0][j];
                q[6] = g[p][6];
                collide7p(q, ep[p], om);
                finish<WHAT>(a, T, q, ep[p], make_float2(fminf(fxy[p].x, f0), fminf(fxy[p].y, f0)), out,
                             src0 >> j & 1u, 1);
                if (own_rows >> j & 1u) {  // (no row of a lane without output columns)
                    if (WHAT != kInside && T.gx + 1 >= a.nx) {  // the column beyond the last
#pragma unroll
                        for (int i = 0; i < 7; i++) q[i].y = 0.f;
                    }
                    ST *o = static_cast<ST *>(a.out) + (out0 + (long long)j * a.pitch);
#pragma unroll
                    for (int i = 0; i < 7; i++) Two<ST>::store(o + i * a.plane + lane, q[i]);
                }
            }
            up = H[j][2];
#pragma unroll
            for (int i = 0; i < 5; i++) H[j][i] = g[p][i];
            H5[0][j] = H5[1][j];
            H5[1][j] = g[p][5];
        }
    }
    sh.edge[par][v][0][T.lane] = H[kRowsZ - 1][2];
    sh.edge[par][v][1][T.lane] = H[0][4];
}

// h_i(x, t) at column x of row r, for the receivers' second time
template <typename ST, bool PER>
__device__ float second_pull(const StepArgs &a, int i, int x, int y, int z) {
    const ST *in = static_cast<const ST *>(a.in);
    const int r = z * a.ny3 + y;
    float g[7];
#pragma unroll
    for (int k = 0; k < 7; k++) {
        int xs = x - Lat<7>::cx(k);
        const int rs = pull_row_yz<7, PER>(a, r, y, z, k);
        if (PER) xs = xs < 0 ? xs + a.nx : xs >= a.nx ? xs - a.nx : xs;
        const bool ok = rs >= 0 && xs >= 0 && xs < a.nx;
        g[k] = ok ? Store<ST>::load1(in + k * a.plane + (long long)rs * a.pitch + xs) : 0.f;
    }
    const float e2 = a.eta2[(long long)r * a.pitch + x];
    collide7(g, e2, a);
    float h = g[0];
#pragma unroll
    for (int k = 1; k < 7; k++)
        if (k == i) h = g[k];
    if (a.src_tab && a.t < a.src_nt && x == a.src_x && r == a.src_y)
        h += (i == 0 ? weight_i<7>(0, e2, a) : weight_i<7>(1, e2, a)) * a.src_tab[a.t];
    if (a.sponge_w > 0) h *= sponge_at<7>(x, r, a);
    return Two<ST>::round(make_float2(h, 0.f)).x;
}

// Receiver r's pressures of both times.  The second state is not in memory: its seven
// populations are computed again from the first (49 loads a receiver, next to a sweep that
// loads 14 values a site).
template <typename ST, bool PER> __device__ void receive(const StepArgs &a, int r) {
    gather_receivers<7, PER, ST>(a, r);
    if (r >= a.nrec || a.trace_row == nullptr) return;
    const int2 xy = a.rec[r];
    const int z = xy.y / a.ny3, y = xy.y - z * a.ny3;
    float rho = 0.f;
#pragma unroll 1
    for (int i = 0; i < 7; i++) {
        int xs = xy.x - Lat<7>::cx(i), ys = y - Lat<7>::cy(i), zs = z - Lat<7>::cz(i);
        if (PER) {
            xs = wrap1(xs, a.nx);
            ys = wrap1(ys, a.ny3);
            zs = wrap1(zs, a.nz);
        } else if (xs < 0 || xs >= a.nx || ys < 0 || ys >= a.ny3 || zs < 0 || zs >= a.nz) {
            continue;
        }
        rho += second_pull<ST, PER>(a, i, xs, ys, zs);
    }
    a.trace_row[a.nrec + (a.rec_col ? a.rec_col[r] : r)] =
        cs2_of<7>(a.eta2[(long long)xy.y * a.pitch + xy.x], a) * rho;
}

template <typename ST>
__global__ void __launch_bounds__(kThreadsZ, 2) sweep3_kernel(const StepArgs a, const SweepArgs w) {
    extern __shared__ __align__(16) unsigned char smem[];
    SharedZ<ST> &sh = *reinterpret_cast<SharedZ<ST> *>(smem);
    asm volatile("griddepcontrol.wait;" ::: "memory");  // (no early launch of dependents: wave.cuh)
    int b = (int)blockIdx.x;
    if (b < w.rec_blocks) {  // block-uniform
        const int r = b * kThreadsZ + (int)threadIdx.x;
        if (w.per)
            receive<ST, true>(a, r);
        else
            receive<ST, false>(a, r);
        return;
    }
    b -= w.rec_blocks;
    const int tiles = w.tx * w.ty, chunk = b / tiles, by = (b - chunk * tiles) / w.tx,
              bx = b - chunk * tiles - by * w.tx,
              v = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    Lane T;
    T.lane = threadIdx.x & 31;
    T.per = w.per != 0;
    const int xlo = bx * w.outx, xhi = min(xlo + w.outx, a.nx);  // output columns
    const int ylo = by * w.outy, yhi = min(ylo + w.outy, a.ny3);
    const int zlo = (int)((long long)a.nz * chunk / w.chunks),
              zhi = (int)((long long)a.nz * (chunk + 1) / w.chunks);
    const int y0 = ylo - kHaloY + v * kRowsZ;
    T.gx = xlo - kHaloX + 2 * T.lane;
    T.gxw = T.gx;
    T.live = T.gx <= xhi + 1;  // level 1 of column xhi pulls from xhi + 1
    if (T.per) {
        T.gxw = wrap1(T.gx, a.nx);  // (nx is even: a lane's columns stay together)
    } else {
        T.live = T.live && T.gx >= 0 && T.gx < a.nx;
    }
    T.own = T.gx >= xlo && T.gx < xhi;
    unsigned rows = 0;  // the warp's rows that level 1 has to compute
#pragma unroll
    for (int j = 0; j < kRowsZ; j++) rows |= y0 + j <= yhi ? 1u << j : 0u;
    unsigned own_rows = 0;  // its output rows, of lanes with output columns
#pragma unroll
    for (int j = 0; j < kRowsZ; j++) own_rows |= T.own && y0 + j >= ylo && y0 + j < yhi ? 1u << j : 0u;
    const int sw = a.sponge_w;
    const bool faces = !T.per || sw > 0;
    const bool gen = faces && (xlo - 1 < sw || xhi >= a.nx - sw || ylo - 1 < sw || yhi >= a.ny3 - sw);
    T.src_cols = 0;
#pragma unroll
    for (int j = 0; j < kRowsZ; j++) {
        const int yw = at_or_none(y0 + j, a.ny3, T.per);
        float f[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int x = at_or_none(T.gx + c, a.nx, T.per);
            const int d = min(min(x, a.nx - 1 - x), min(yw, a.ny3 - 1 - yw));
            f[c] = x < 0 || yw < 0 ? -1.f : sw > 0 ? sponge_of_dist(d, a) : 1.f;
            if (x == a.src_x) T.src_cols |= 1u << c;
        }
        sh.factor[v * kRowsZ + j][T.lane] = make_float2(f[0], f[1]);
        sh.e2[v * kRowsZ + j][T.lane] = f2(0.f);
    }
    unsigned src_rows = 0;
    if (a.src_tab != nullptr && a.t < a.src_nt && __any_sync(0xffffffffu, T.src_cols != 0)) {
#pragma unroll
        for (int j = 0; j < kRowsZ; j++)
            if (at_or_none(y0 + j, a.ny3, T.per) == a.src_y % a.ny3) src_rows |= 1u << j;
    }
    if (threadIdx.x < 256) sh.tab[threadIdx.x] = a.mid ? a.mid_tab[threadIdx.x] : 0.f;
    float2 H[kRowsZ][5], H5[2][kRowsZ];
#pragma unroll
    for (int j = 0; j < kRowsZ; j++) {
        H5[0][j] = H5[1][j] = f2(0.f);
#pragma unroll
        for (int i = 0; i < 5; i++) H[j][i] = f2(0.f);
    }
    const int sz = a.src_y / a.ny3;
    const int lane = T.gx;               // the lane's columns in a row
    const int from = T.live ? lane : 0;  // where it copies from (nothing if not live)
    // rows inside with those next to them (the rows beyond the tile's are copied too)
    const bool rows_in = y0 >= 1 && y0 + kRowsZ < a.ny3;
    const bool whole = !T.per || (rows_in && !__any_sync(0xffffffffu, T.gx != T.gxw));
    const bool out = !T.per && (xlo == 0 || xhi >= a.nx || ylo == 0 || yhi >= a.ny3);
    const bool pad = xhi == a.nx && (a.nx & 1) != 0;
#pragma unroll 1
    for (int z = zlo - 2; z <= zhi; z++) {
        const bool planes_in = z >= 0 && z + 2 < a.nz;  // plane z + 1 and its neighbours
        const bool next = whole && (!T.per || planes_in);  // without the general copies
        if (z >= zlo - 1) {
            __syncthreads();  // the edges of plane z - 1, and (first) the table
            bool edge = gen || pad || (!T.per && !(rows_in && planes_in));
            if (faces) edge = edge || z - 1 < sw || z >= a.nz - sw;
            unsigned s1 = 0, s0 = 0;
            if (src_rows) {
                s1 = at_or_none(z, a.nz, T.per) == sz ? src_rows : 0u;
                s0 = at_or_none(z - 1, a.nz, T.per) == sz ? src_rows : 0u;
            }
            const bool ghost = out || (!T.per && (z - 1 < 0 || z >= a.nz));
            // the warp's first row in planes z + 1 and z - 1
            const long long up0 = row_start(y0, z + 1, a.ny3, a.pitch),
                            down0 = row_start(y0, z - 1, a.ny3, a.pitch);
            if (rows == 0) {  // warp-uniform
            } else if (edge || (s1 | s0))
                plane<ST, kEdges>(a, T, sh, H, H5, v, y0, z, next && z < zhi, up0, from, z - 1 >= zlo,
                                  down0, lane, own_rows, ghost, s1, s0);
            else
                plane<ST, kInside>(a, T, sh, H, H5, v, y0, z, next && z < zhi, up0, from, z - 1 >= zlo,
                                   down0, lane, own_rows, false, 0u, 0u);
        }
        if (rows && z < zhi && !(next && z >= zlo - 1)) {
#pragma unroll 1
            for (int j = 0; j < kRowsZ; j++) {
                issue<ST>(a, T, sh, v * kRowsZ + j, y0 + j, z + 1, rows >> j & 1u);
                if (j % kTake == kTake - 1) cp_commit();  // (the groups that plane() waits for)
            }
        }
    }
}

}  // namespace lbsweep3
