// wave.cu -- host side of the warp wavefront (kernels: wave.cuh): FP32 D2Q5 instances, the
// choice of steps per launch and of the launch shape, receiver row lists and served batches.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "lb_kernels.cuh"
#include "lb_runtime.h"
#include "tile.cuh"
#include "wave.cuh"
#include "wave_host.h"

using namespace lbk;
using namespace lbrt;
using namespace lbwave;
using namespace lbtile;

namespace lbwave {
WavePick pick_d2q5_f32(int ck, int K, bool rec, bool per) {
    if (K == 6)  // BGK only (wave_steps)
        return ck == kLossless ? rec ? pick_one<5, kLossless, 6, true, float, false>(per)
                                     : pick_one<5, kLossless, 6, false, float, false>(per)
                               : rec ? pick_one<5, kBgk, 6, true, float, false>(per)
                                     : pick_one<5, kBgk, 6, false, float, false>(per);
    return K == 4 ? pick_rec<5, 4, float, false>(ck, rec, per) : pick_rec<5, 2, float, false>(ck, rec, per);
}
WaveBatchFn pick_batch_fp32(bool mrt, bool per) { return pick_batch<false>(mrt, per); }
}  // namespace lbwave

namespace lbrt {
int sm_count() {
    static std::atomic<int> sms{0};
    int v = sms.load(std::memory_order_relaxed);
    if (!v) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            v = 1;
        }
        sms.store(v, std::memory_order_relaxed);
    }
    return v;
}

}  // namespace lbrt

namespace {

int collision_kind(const lb_ctx *c) {
    if (c->cfg.collision == LB_MRT) return kMrt;
    return c->Q == 5 && (float)(1.0 / c->cfg.tau) == 2.f ? kLossless : kBgk;
}

WavePick pick(const lb_ctx *c, int K, bool rec) {
    const int ck = collision_kind(c);
    const bool per = c->cfg.boundary == LB_PERIODIC;
    if (c->Q == 9)
        return c->cfg.storage == LB_BF16 ? pick_d2q9_bf16(ck, K, rec, per)
                                         : pick_d2q9_f32(ck, K, rec, per);
    if (c->cfg.storage == LB_F16) return pick_d2q5_f16(ck, rec, per);
    return c->cfg.storage == LB_BF16 ? pick_d2q5_bf16(ck, K, rec, per) : pick_d2q5_f32(ck, K, rec, per);
}

// What a row in the sponge or of a strip at a face counts against kInner: an iteration with sponge
// factors issues half as many instructions again, one with the cuts at a zero-ghost face (wave.cuh)
// more.  Times of 85 zero-ghost grids of 0.2 to 25 million sites at weights of 8 / 9 / 10 / 11 / 12 / 13 / 14
// sixths against the best: with a sponge D2Q5 FP32 1.06 / 1.03 / 1.01 / 1.01 / 1.01 / 1.00 / 1.00, BF16 1.06 /
// 1.04 / 1.03 / 1.01 / 1.00 / 1.00 / 1.00, D2Q9 BF16 1.06 / 1.02 / 1.00 / 1.00 / 1.00 / 1.01 / 1.01, FP32
// 1.12 / 1.08 / 1.03 / 1.01 / 1.00 / 1.00 / 1.00; without D2Q5 BF16 1.00 / 1.01 / 1.02 / 1.02 / 1.03 / 1.04 / 1.03,
// the others about as with; six steps without a sponge 2779 x 8574 1.34 / 1.24 / 1.18 / 1.13 / 1.08 / 1.03 / 1.00.
// Periodic grids cut nothing: 4/3 where the four-step FP32 BGK launch waits for HBM in part, 3/2
// elsewhere.
int outer_weight(const lb_ctx *c, int K) {
    if (c->cfg.boundary != LB_PERIODIC) {
        if (c->Q == 9) return 12;
        if (c->cfg.sponge_width > 0) return 13;
        return K == 6 ? 14 : c->cfg.storage == LB_BF16 ? 9 : 12;
    }
    return c->Q == 5 && K <= 4 && c->cfg.storage == LB_F32 && c->cfg.collision == LB_BGK ? 8 : 9;
}

// Strips, and which of them meet the sponge or a face.  Strip b takes columns b out - halo ..
// b out - halo + kCols - 1, recomputed ones included.
void strips_of(WaveArgs &w, int nx, int K, int sponge, bool per) {
    const int out = out_cols(K);
    w.per = per ? 1 : 0;
    w.strips = (nx + out - 1) / out;
    w.edge_l = w.edge_r = 0;
    if (!per || sponge > 0 || nx % 2) {
        w.edge_l = std::min(w.strips, (sponge + halo(K) + out - 1) / out);
        const int first = std::max(0, nx - sponge - (kCols - halo(K)) + out) / out;
        w.edge_r = w.strips - std::min(w.strips, std::max(w.edge_l, first));
    }
}

// n row chunks for the inner strips; returns the tasks
long long set_chunks(WaveArgs &w, int ny, long long n) {
    const int edge = w.edge_l + w.edge_r;
    w.chunks = (int)n;
    w.chunks_e = (int)std::min<long long>(ny, (w.outer * n + kInner - 1) / kInner);
    const long long t = (long long)(w.strips - edge) * w.chunks + (long long)edge * w.chunks_e;
    w.tasks = (int)t;
    return t;
}

// Row chunks of a grid.  A warp sweeps its H + 2K rows one after another, of which 2K are
// recomputed, so few tall chunks waste little and many short ones finish sooner while warps are
// missing.  With m warps per scheduler an iteration of all of them takes about (4 + m) x 0.12 us
// (K = 4, GB300: 0.57, 0.67, 0.82 and 0.96 us for m = 1 .. 4 at 4096^2, 0.66 .. 1.0 at 512^2);
// the m that makes (H + 2K)(4 + m) smallest wins, and its tasks fit one wave.
void shape(WaveArgs &w, int ny, int K, int max_m) {
    const long long slots1 = (long long)sm_count() * kWarpsPerCta;
    long long cost = -1, best = 1;
    for (int m = 1; m <= max_m; m++) {
        long long n = std::max<long long>(1, std::min<long long>(ny, m * slots1 / w.strips));
        while (n > 1 && set_chunks(w, ny, n) > m * slots1) n--;
        const long long c = ((ny + n - 1) / n + 2 * K) * (4 + m);
        if (cost < 0 || c < cost) cost = c, best = n;
    }
    set_chunks(w, ny, best);
}

}  // namespace

bool wave_supported(const lb_ctx *c) {
    return (c->Q == 5 || c->Q == 9) && c->nz <= 1 && !c->refined && !c->aa && !c->slab_nyg &&
           (c->cfg.storage == LB_F32 || c->cfg.storage == LB_BF16 ||
            (c->cfg.storage == LB_F16 && c->Q == 5));
}

// A launch of four steps takes about 10 us however small the grid is, and longer with receivers;
// a step alone takes 3 (128^2: 3.5 us a step fused against 3.0; 512^2: 4.6 against 5.4).
static bool wave_pays(const lb_ctx *c) { return (long long)c->ny * c->pitch >= (128LL << 10); }

// Six steps (three CTAs per SM) beat four (four CTAs) where HBM is the limit: FP32 BGK grids well
// beyond L2 (8192^2: 645 GLUPS against 560, 3000 x 2500: 470 against 440; 2048^2, 168 MB: 379
// against 388).  MRT and BF16 are bound by issue first and run four (4096^2 MRT: 525 against
// 470, BF16: 541 against 493).
static int wave_steps(const lb_ctx *c, int n) {
    if (c->Q == 5 && c->cfg.storage == LB_F32 && c->cfg.collision == LB_BGK && n >= 6 && n != 8 &&
        2LL * 5 * 4 * c->ny * c->pitch >= (200LL << 20))
        return 6;
    // D2Q9 BF16: four steps on large grids, two on small ones (4096^2: 261 against 229 GLUPS,
    // 2048^2: 192 against 198, 512^2: 46 against 54); FP32: four (4096^2: 264 against 165)
    if (c->Q == 9 && c->cfg.storage == LB_BF16 && (long long)c->ny * c->pitch < (6LL << 20))
        return n >= 2 ? 2 : 1;
    return n >= 4 ? 4 : n >= 2 ? 2 : 1;
}

// Per-row receiver lists (rows of the context, x ascending), one allocation.
lb_status wave_set_receivers(lb_ctx *ctx, const int *xy, int nrec) {
    if (ctx->row_off) dev_free(ctx, ctx->row_off);
    ctx->row_off = ctx->row_x = ctx->row_id = ctx->row_y = nullptr;
    const size_t no = (size_t)ctx->ny + 2, nr = (size_t)std::max(nrec, 1);
    std::vector<int> all(no + 3 * nr, 0);
    int *off = all.data(), *xs = off + no, *ids = xs + nr, *ys = ids + nr;
    for (int r = 0; r < nrec; r++) off[(size_t)xy[2 * r + 1] + 1]++;
    for (size_t k = 1; k < no; k++) off[k] += off[k - 1];
    for (int r = 0; r < nrec; r++) ids[r] = r;
    std::stable_sort(ids, ids + nrec, [&](int p, int q) {
        return xy[2 * p + 1] != xy[2 * q + 1] ? xy[2 * p + 1] < xy[2 * q + 1] : xy[2 * p] < xy[2 * q];
    });
    for (int k = 0; k < nrec; k++) xs[k] = xy[2 * ids[k]], ys[k] = xy[2 * ids[k] + 1];
    int *d = static_cast<int *>(dev_alloc(ctx, all.size() * sizeof(int)));
    if (!d) return fail(ctx, LB_ENOMEM, "row receiver lists");
    cudaError_t e = cudaMemcpyAsync(d, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice,
                                    ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);  // `all` goes out of scope
    ctx->row_off = d;
    ctx->row_x = d + no;
    ctx->row_id = ctx->row_x + nr;
    ctx->row_y = ctx->row_id + nr;
    if (e != cudaSuccess) return cuda_fail(ctx, e, "row receiver lists");
    return LB_OK;
}

static lb_status wave_launch(lb_ctx *ctx, const StepArgs &a, WaveArgs w, int K) {
    const WavePick p = pick(ctx, K, a.rho_out != nullptr);
    w.outer = outer_weight(ctx, K);
    strips_of(w, ctx->nx, K, a.sponge_w, ctx->cfg.boundary == LB_PERIODIC);
    shape(w, ctx->ny, K, p.ctas);
    cudaError_t e = cudaFuncSetAttribute(p.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "wavefront shared memory");
    e = launch_pdl(p.fn, dim3((w.tasks + kWarpsPerCta - 1) / kWarpsPerCta), dim3(kCtaThreads), p.smem,
                   ctx->stream, a, w);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "wavefront launch");
    return LB_OK;
}

// tiles of K steps, and how many to a row of tiles
static int tiles_of(const lb_ctx *c, int K, int *tx) {
    const int ox = kSide - 2 * halo_x(K), oy = kSide - 2 * K;
    *tx = (c->nx + ox - 1) / ox;
    return *tx * ((c->ny + oy - 1) / oy);
}

static lb_status tile_launch(lb_ctx *ctx, const StepArgs &a, const WaveArgs &rec, int K) {
    TileArgs t;
    t.rec = rec;
    t.K = K;
    const int tiles = tiles_of(ctx, K, &t.tx), ctas = tiles <= sm_count() ? 1 : 2;
    const int ck = collision_kind(ctx);
    const bool rho = a.rho_out != nullptr, per = ctx->cfg.boundary == LB_PERIODIC;
    const TileFn fn = ctx->cfg.storage == LB_BF16 ? pick_tile_bf16(ck, rho, ctas, per)
                                                  : pick_tile_f32(ck, rho, ctas, per);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Shared));
    if (e == cudaSuccess)
        e = launch_pdl(fn, dim3(tiles), dim3(kTileThreads), sizeof(Shared),
                       ctx->stream, a, t);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "tile launch");
    return LB_OK;
}

// f.steps fused steps with the caller's arguments (a.in must not be raw); receivers when
// a.trace_row is set and the row lists exist; rho of every level when a.rho_out is set.
lb_status fuse_launch_args(lb_ctx *ctx, const StepArgs &a, Fuse f) {
    if (ctx->Q == 7) return sweep3_launch(ctx, a);
    WaveArgs w = {};
    w.row_off = a.trace_row ? ctx->row_off : nullptr;
    w.rec_x = ctx->row_x;
    w.rec_id = ctx->row_id;
    w.rec_y = ctx->row_y;
    w.per = ctx->cfg.boundary == LB_PERIODIC ? 1 : 0;
    return f.tile ? tile_launch(ctx, a, w, f.steps) : wave_launch(ctx, a, w, f.steps);
}

// About what a launch of K steps on tiles takes, in 0.01 us, from GB300 times of 128^2 to 2048^2
// grids for K = 4 .. 16: with q tiles per SM, 5.2 + 0.54 K us up to one, then the larger of
// 6 + 1.35 K (two share an SM) and 4 + q (2.5 + 0.62 K).
static long long tile_cost(const lb_ctx *c, int K) {
    int tx;
    const long long t = tiles_of(c, K, &tx), sms = sm_count();
    if (t <= sms) return 520 + 54 * K;
    return std::max<long long>(600 + 135 * K, 400 + t * (250 + 62 * K) / sms);
}

// The next launch of n wanted steps.  D2Q5 grids up to 3.5 million sites go on tiles, in launches
// of the K <= 16 steps that cost least each (evened out over the launches that n takes), where
// that beats single steps of about 3.1 us + 6 ps a site; above, and for D2Q9, the wavefront is
// faster (2048^2: 10.8 against 11.0 us a step, 4096^2: 29 against 44).
Fuse fuse_steps(const lb_ctx *c, int n) {
    const long long sites = (long long)c->ny * c->pitch;
    if (c->Q == 7) return Fuse{n >= 2 && sweep3_pays(c) ? 2 : 1, false};
    // FP16: two, since its range scales are guessed no further ahead (a launch, the scale update and
    // a second launch that mostly ends at once; 3001 x 1777: 25.5 us a step against 35.9).  They pay
    // against the staged step (1420 x 675: 12.1 against 17.0), not against the register-streaming one
    // of narrower grids (431 x 1307: 11.4 against 9.1).
    // At the seam of odd periodic rows a 16-bit wavefront copies value by value, while the other strips
    // wait (FP16 1471 x 3767: 57 us a step against 38; BF16 4017 x 3861: 88 against 63).
    const bool seam = c->cfg.boundary == LB_PERIODIC && c->nx % 2 != 0;
    if (c->cfg.storage == LB_F16)
        return Fuse{n >= 2 && c->staged && sites >= 500000 && !seam ? 2 : 1, false};
    if (c->Q == 5 && sites < 3500000) {
        // two steps alone: a launch of tiles takes 8 us however few they are (614 x 117 periodic: 4.2 us a
        // step against 2.9, 991 x 996: 6.0 against 5.4; three: 2.9 against 2.9)
        if (n < 2 || (n == 2 && c->cfg.time_block <= 1)) return Fuse{1, false};
        int best = 2;
        long long cost = -1;
        for (int K = 2; K <= 16; K += 2) {
            const long long x = tile_cost(c, K);
            if (cost < 0 || x * best < cost * K) cost = x, best = K;
        }
        const int launches = (n + best - 1) / best, K = (n + launches - 1) / launches;
        if (tile_cost(c, K) >= K * (310 + sites * 6 / 10000)) return Fuse{1, false};
        return Fuse{K, true};
    }
    if (seam && c->cfg.storage == LB_BF16) return Fuse{1, false};
    if (c->cfg.time_block <= 1) {
        if (!wave_pays(c)) return Fuse{1, false};
        // D2Q9 FP32 grids below a million sites run one step as fast in L2 (708 x 739 MRT: 8.7 us
        // against 9.9, 374 x 3184: 16.6 against 13.9), odd periodic ones below two (297 x 4006: 15.2
        // against 16.2, 1183 x 1183 in threes 15.9 against 17.2; 1415 x 1413: 25.8 against 20.4)
        if (c->Q == 9 && c->cfg.storage == LB_F32 && sites < (seam ? 1800000 : 1000000))
            return Fuse{1, false};
        // two steps at a time: odd periodic D2Q5 grids of less than 5.4 million sites (1923 x 1924: 23.7
        // against 25.0, 2345 x 2345: 35.3 against 32.9)
        if (c->Q == 5 && seam && n < 4 && sites < 5400000) return Fuse{1, false};
    }
    return Fuse{wave_steps(c, n), false};
}

// ---------------------------------------------------------------- fused launches --
// cfg.time_block values (fuse_steps takes them in launches that suit)
bool tb_supported(int Q, int K) {
    return Q == 5 ? K == 2 || K == 4 || K == 6 || K == 8 || K == 16 : K == 2 || K == 4;
}

// K fused steps of the context from a non-raw state; the caller keeps them inside the trace
// buffer and the rho tape.
lb_status tb_launch(lb_ctx *ctx, Fuse f) {
    const int K = f.steps;
    StepArgs a = base_args(ctx);
    a.in = ctx->pop[ctx->cur];
    a.out = ctx->pop[ctx->cur ^ 1];
    a.t = ctx->t;
    a.raw = 0;
    const long long row = ctx->t - ctx->t_rec0;
    a.trace_row = (ctx->trace && (ctx->row_off || ctx->Q == 7) && row >= 0 && row + K <= ctx->trace_cap)
                      ? ctx->trace + row * ctx->nrec : nullptr;
    a.rho_out = tape_row(ctx, ctx->t);  // level j at rho_out + j plane
    a.rho_stride = (long long)ctx->ny * ctx->pitch;
    if (ctx->lp_scale) f16_slots(ctx, a, K);
    lb_status st = ctx->cfg.storage == LB_BF16 && ctx->cfg.time_block > 1
                       ? tb5_launch_args(ctx, a, K)
                       : fuse_launch_args(ctx, a, f);
    if (st == LB_OK && ctx->lp_scale && (st = f16_update(ctx, a)) == LB_OK) {
        a.redo = f16_redo(ctx);  // once more, where the second step's scale was another
        ctx->n_launch++;
        st = fuse_launch_args(ctx, a, f);
    }
    if (st != LB_OK) return st;
    ctx->cur ^= 1;
    ctx->t += K;
    return LB_OK;
}

// ------------------------------------------------------------- served batches --
// One launch of wave_batch_kernel: the descriptors of its n shots in one staging block,
// [n] StepArgs, [n] WaveArgs, [n + 1] block prefixes.
namespace {
size_t up256(size_t v) { return (v + 255) / 256 * 256; }
struct BatchLayout {
    StepArgs *a;
    WaveArgs *w;
    int *first;
};
BatchLayout batch_layout(void *base, int n) {
    char *p = static_cast<char *>(base);
    BatchLayout L;
    L.a = reinterpret_cast<StepArgs *>(p);
    p += up256(n * sizeof(StepArgs));
    L.w = reinterpret_cast<WaveArgs *>(p);
    p += up256(n * sizeof(WaveArgs));
    L.first = reinterpret_cast<int *>(p);
    return L;
}
// tasks and shape of one shot at about H rows per chunk
int batch_shape(const lb_ctx *c, int H, WaveArgs &w) {
    // (9 sixths on small shots, whose chunks are short already: 32 of 256^2 568 shots/s against 461 at
    // 10, of 2048^2 37.8 against 38.7 at 11)
    w.outer = c->ny < 1024 ? 9 : 11;
    strips_of(w, c->nx, kServeSteps, c->cfg.sponge_width, c->cfg.boundary == LB_PERIODIC);
    H = std::max(1, std::min(c->ny, H));
    return (int)set_chunks(w, c->ny, (c->ny + H - 1) / H);
}
int ctas_of(int tasks) { return (tasks + kWarpsPerCta - 1) / kWarpsPerCta; }
}  // namespace

size_t wave_batch_bytes(int n) {
    return up256(n * sizeof(StepArgs)) + up256(n * sizeof(WaveArgs)) + up256((n + 1) * sizeof(int));
}

bool wave_batch_ready(const lb_ctx *ctx) {
    constexpr int K = kServeSteps;
    if (ctx->Q != 5 || ctx->cfg.storage == LB_F16 || !wave_supported(ctx) || ctx->raw || ctx->ckpt_every > 0) return false;
    if (ctx->rho_tape) {
        const long long row = ctx->t - ctx->tape_t0;
        if (row < 0 || row + K > ctx->tape_cap) return false;
    }
    if (ctx->nrec > 0) {
        const long long row = ctx->t - ctx->t_rec0;
        if (!ctx->row_off || row < 0 || row + K > ctx->trace_cap) return false;
    }
    return true;
}

int wave_batch_rows(lb_ctx *const *ctxs, int n) {
    // the rows per warp of shape(), over all shots' strips
    long long rows = 0;
    int ny = 1;
    for (int k = 0; k < n; k++) {
        WaveArgs w;
        strips_of(w, ctxs[k]->nx, kServeSteps, ctxs[k]->cfg.sponge_width, false);
        rows += (long long)w.strips * ctxs[k]->ny;
        ny = std::max(ny, ctxs[k]->ny);
    }
    const long long slots1 = (long long)sm_count() * kWarpsPerCta;
    long long cost = -1, best = 1;
    for (int m = 1; m <= 2; m++) {  // (three: 512^2 291 shots/s against 357, 2048^2 35.5 against 37.8)
        const long long H = std::min<long long>(ny, (rows + m * slots1 - 1) / (m * slots1));
        const long long c = (H + 2 * kServeSteps) * (4 + m);
        if (cost < 0 || c < cost) cost = c, best = H;
    }
    return (int)best;
}

bool wave_batch_round(lb_ctx *const *ctxs, int n) {
    static std::atomic<int> l2{-1};
    int bytes = l2.load(std::memory_order_relaxed);
    if (bytes < 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&bytes, cudaDevAttrL2CacheSize, dev) != cudaSuccess) {
            cudaGetLastError();
            bytes = 0;
        }
        l2.store(bytes, std::memory_order_relaxed);
    }
    long long rows = 0, state = 0;
    for (int k = 0; k < n; k++) {
        rows += (long long)((ctxs[k]->nx + 247) / 248) * ctxs[k]->ny;
        state += 2LL * ctxs[k]->Q * ctxs[k]->ny * ctxs[k]->pitch * ctxs[k]->ebytes;
    }
    return !(rows > 11LL * 3 * sm_count() && 4 * state > 3LL * bytes);
}

int wave_batch_blocks(const lb_ctx *ctx, int H) {
    WaveArgs w;
    return ctas_of(batch_shape(ctx, H, w));
}

// Fill the host staging block `h` for kServeSteps steps of ctxs[0 .. n), about H output rows per
// warp (advancing their time and buffers as if the launch ran); returns the block count.
int wave_batch_fill(lb_ctx *const *ctxs, int n, int H, void *h) {
    BatchLayout L = batch_layout(h, n);
    int blocks = 0;
    for (int k = 0; k < n; k++) {
        lb_ctx *ctx = ctxs[k];
        StepArgs a = base_args(ctx);
        a.in = ctx->pop[ctx->cur];
        a.out = ctx->pop[ctx->cur ^ 1];
        a.t = ctx->t;
        a.raw = 0;
        a.rho_out = tape_row(ctx, ctx->t);
        a.rho_stride = (long long)ctx->ny * ctx->pitch;
        const long long row = ctx->t - ctx->t_rec0;
        a.trace_row = ctx->nrec > 0 ? ctx->trace + row * ctx->nrec : nullptr;
        WaveArgs w;
        w.row_off = a.trace_row ? ctx->row_off : nullptr;
        w.rec_x = ctx->row_x;
        w.rec_id = ctx->row_id;
        w.rec_y = ctx->row_y;
        w.bf16 = ctx->cfg.storage == LB_BF16 ? 1 : 0;
        const int tasks = batch_shape(ctx, H, w);
        L.a[k] = a;
        L.w[k] = w;
        L.first[k] = blocks;
        blocks += ctas_of(tasks);
        ctx->cur ^= 1;
        ctx->t += kServeSteps;
    }
    L.first[n] = blocks;
    return blocks;
}

cudaError_t wave_batch_launch(const void *d, int n, int blocks, bool mrt, bool round,
                              bool per, cudaStream_t stream) {
    if (n < 1 || blocks < 1) return cudaErrorInvalidValue;
    const WaveBatchFn fn = round ? pick_batch_round(mrt, per) : pick_batch_fp32(mrt, per);
    constexpr int smem = cta_bytes<5, kServeSteps, float>();
    static_assert(smem >= cta_bytes<5, kServeSteps, __nv_bfloat16>(), "room for either storage");
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    BatchLayout L = batch_layout(const_cast<void *>(d), n);
    return launch_pdl(fn, dim3(blocks), dim3(kCtaThreads), smem, stream, (const StepArgs *)L.a,
                      (const WaveArgs *)L.w, (const int *)L.first, n);
}
