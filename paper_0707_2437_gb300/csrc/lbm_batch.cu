// Host side of the batched form (the kernels are in lbm_batch_kernels.cuh):
// many uneven grids (any size, tau, c2 and storage) advanced by persistent kernels over a
// tile work-list, replayed from a CUDA graph: one cooperative launch per kind group with
// a grid-wide barrier between passes (lockstep), or one launch with progress counters per
// tile (flow).  This file plans: which kernel each group runs, whether its passes take
// one, two or three steps, how tall its tiles are.
//
// Every barrier wait is bounded (wall-clock limit read from %globaltimer): a
// block that gives up sets a status word and returns, all other blocks see the
// status at their next barrier and return too, so the kernel always ends.
#include <algorithm>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_internal.h"
#include "lbm_batch_kernels.cuh"

struct lbm_batch {
    std::vector<lbm_grid *> grids;
    cudaStream_t stream = nullptr;
    int device = 0;
    int rows = 16;
    bool fit_rows = true;   // default: lockstep work-lists may use shorter tiles
    int blocks_per_sm = 0;  // 0: the occupancy limit
    // Kind groups: consecutive ranges of the tile list, each run by its own
    // persistent launch (a specialised k_batch_one, or k_batch for the rest),
    // one after the other on the batch's stream.
    struct Group {
        int begin = 0, count = 0;
        BatchKernel kernel = nullptr;
        FlowKernel fkernel = nullptr;  // flow schedule
        int smem = 0;                  // dynamic shared memory per block
        bool fused = false;            // several steps per pass (the fused walk)
        int rows = 0;                  // tile height
        int max_blocks_per_sm = 1;
    };
    // A work-list: the grids' records and tiles on the device, the groups that run them.
    struct List {
        std::vector<Group> groups;
        GridDesc *d_grids = nullptr;
        Tile *d_tiles = nullptr;
        int ntiles = 0;
        int paired = 0;        // tiles with two segments (split walk)
        std::vector<int> per;  // per grid, the steps of its passes
        // graph cache (one step count)
        cudaGraphExec_t graph = nullptr;
        long long graph_n = -1;
        // The list on the device is the one of the batch's settings.  A build that fails
        // leaves none, and the next step call builds again before it launches anything;
        // so does one that finds another c2 field or rounding than the list was built for.
        bool built = false;
        std::vector<const float *> built_a15f;
        std::vector<int> built_rounding;
    };
    // The list of step calls, and one of single-step walks for calls of one step where
    // the first takes several a pass, made by the first such call: a pass cut to one step
    // reads the halo of several and walks narrower strips (one step of nine 2048^2 grids
    // FP32 545 us in such a pass, 417 in single steps; FP16 291 / 236).
    List list[2];
    int walk16 = LBM_WALK16_AUTO;  // walk of 16-bit grids (lbm_batch_set_walk16)
    int sms = 1;
    unsigned long long timeout_ns = 1000000000ULL;
    // device
    long long *d_limit = nullptr;
    int *d_parity = nullptr;
    uint32_t *d_t0 = nullptr;
    unsigned *d_bar = nullptr;
    int *d_status = nullptr;
    // pinned host mirrors of the per-call arrays
    long long *h_limit = nullptr;
    int *h_parity = nullptr;
    uint32_t *h_t0 = nullptr;
    int *h_status = nullptr;
    cudaEvent_t copied = nullptr;  // the per-call arrays have been read
    // Streams of members other than the batch's own (as of the last step
    // call), with one event each, and the event that marks the batch's work.
    std::vector<cudaStream_t> xs;
    std::vector<cudaEvent_t> xev;
    cudaEvent_t done = nullptr;
    // Launch mode (lbm_batch_set_launch): LBM_LAUNCH_AUTO tries a graph and
    // falls back to direct launches if capture fails, LBM_LAUNCH_GRAPH
    // requires the graph, LBM_LAUNCH_DIRECT never captures.  `capture_failed`
    // records an AUTO fallback; `last_launch` is how the last step call ran
    // (0 before the first one).
    int launch_mode = LBM_LAUNCH_AUTO;
    bool capture_failed = false;
    int last_launch = 0;
    // Schedule (lbm_batch_set_schedule): lockstep kind groups, or one flow
    // launch over all grids with per-tile progress (control words per grid,
    // completed steps per tile, and the count of grids with work this call).
    int schedule = LBM_SCHEDULE_LOCKSTEP;
    unsigned long long *d_ctl = nullptr;
    int *d_prog = nullptr;
    size_t prog_cap = 0;
    int *d_nwork = nullptr;
    int *h_nwork = nullptr;
};

static int bfail(int code, const std::string &m) {
    set_error(m);
    return code;
}

static int bcuda(cudaError_t e, const char *where) {
    set_error(std::string(where) + ": " + cudaGetErrorString(e));
    cudaGetLastError();  // reported here: a later launch does not meet it again
    return e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
}

#define BCK(call)                                           \
    do {                                                    \
        cudaError_t e_ = (call);                            \
        if (e_ != cudaSuccess) return bcuda(e_, #call);     \
    } while (0)

static void drop_graph(lbm_batch::List &w) {
    if (w.graph) cudaGraphExecDestroy(w.graph);
    w.graph = nullptr;
    w.graph_n = -1;
}
static void drop_graphs(lbm_batch *b) {
    for (lbm_batch::List &w : b->list) drop_graph(w);
}

// Sites per lane of a grid's walk.  FP32: 4 (128-bit loads) when nx is a
// multiple of 4.  16-bit: 8 (128-bit loads, rows and any c2 field's values
// through shared memory) when nx is a multiple of 8 and the walk is
// LBM_WALK16_AUTO or LBM_WALK16_V8; else 4 (64-bit loads, one row prefetched
// in registers) when nx is a multiple of 4.  Any other nx: 1.  (Measured on GB300: 8 sites
// per lane run 15 % faster than 4 with nearest rounding and 10 % faster with
// stochastic rounding.)
static int batch_vec(const lbm_batch *b, const lbm_grid *g) {
    const bool eight = b->walk16 == LBM_WALK16_V8 || b->walk16 == LBM_WALK16_AUTO;
    if (g->storage != ST_F32 && eight && g->nx % 8 == 0) return 8;
    return g->nx % 4 == 0 ? 4 : 1;
}

// Copies the grid table and the tile list to the device.
static int upload_worklist(lbm_batch *b, lbm_batch::List &w, const std::vector<GridDesc> &gd,
                           const std::vector<Tile> &ordered) {
    if (w.d_tiles) cudaFree(w.d_tiles);
    w.d_tiles = nullptr;
    BCK(cudaMalloc(&w.d_tiles, sizeof(Tile) * std::max<size_t>(1, ordered.size())));
    if (!w.d_grids) BCK(cudaMalloc(&w.d_grids, sizeof(GridDesc) * gd.size()));
    BCK(cudaMemcpy(w.d_grids, gd.data(), sizeof(GridDesc) * gd.size(), cudaMemcpyHostToDevice));
    BCK(cudaMemcpy(w.d_tiles, ordered.data(), sizeof(Tile) * ordered.size(),
                   cudaMemcpyHostToDevice));
    w.ntiles = (int)ordered.size();
    w.built_a15f.clear();
    w.built_rounding.clear();
    for (const lbm_grid *g : b->grids) {
        w.built_a15f.push_back(g->a15f);
        w.built_rounding.push_back(g->rounding);
    }
    w.built = true;
    return LBM_OK;
}

// Resident blocks per SM of a kernel of this file, at least one.
static int resident_blocks(const lbm_batch *b, const void *fn, int smem, int *blocks) {
    *blocks = (int)(resident_warps(fn, kBatchWarps, smem) / kBatchWarps / b->sms);
    if (*blocks >= 1) return LBM_OK;
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? bcuda(e, "occupancy of a batch kernel")
                            : bfail(LBM_ECUDA, "batch kernel cannot be resident");
}

// Tile height of a lockstep group on the fused walk, from the grids' strips and
// rows: a tile costs some row steps beyond its rows.  With tiles of one height a
// pass lasts ceil(tiles / warps) of them; in general the warps, which take tiles as
// they finish others, are done within the mean plus one tile.  The lower of both
// bounds decides.
// `fixed`: a height of the caller's (0: the best up to `most`).  *cost: row steps of
// a pass.
static int fused_rows(const std::vector<std::pair<FusedStrips, int>> &grids, long long warps,
                      int overhead, int most, int fixed, double *cost) {
    int rows = 2;
    for (int r = fixed ? fixed : 2; r <= (fixed ? fixed : most); r += r < 64 ? 1 : 4) {
        long long tiles = 0, work = 0;
        int tallest = 0;
        for (const auto &g : grids) {  // (strips, rows)
            const long long segs = (g.second + r - 1) / r, n = g.first.tiles(segs);
            const int high = std::min(r, g.second);
            tiles += n;
            work += n * overhead + g.first.full * g.second + (n - g.first.full * segs) * high;
            tallest = std::max(tallest, high);
        }
        const double even = (double)((tiles + warps - 1) / warps) * (tallest + overhead);
        const double mixed = (double)work / warps + (tallest + overhead);
        const double now = std::min(even, mixed);
        if (*cost == 0 || now < *cost) {
            *cost = now;
            rows = r;
        }
        if (tallest < r) break;  // every grid is one segment
    }
    return rows;
}

// (Re)builds a work-list; singles_only: of single-step walks.
static int build_list(lbm_batch *b, lbm_batch::List &w, bool singles_only) {
    w.built = false;
    drop_graph(w);  // (it launches on the old list)
    const size_t ng = b->grids.size();
    std::vector<GridDesc> gd(ng);
    std::vector<Tile> tiles;
    w.paired = 0;
    w.per.assign(ng, 1);
    w.groups.clear();
    bool slabs = false;
    for (size_t k = 0; k < ng; ++k) {
        lbm_grid *g = b->grids[k];
        GridDesc &d = gd[k];
        d.buf[0] = g->buf[0];
        d.buf[1] = g->buf[1];
        d.a15f = g->a15f;
        d.P = g->P;
        d.nx = g->nx;
        d.ny = g->ny;
        d.kind = kind_code(g->storage, batch_vec(b, g), g->rounding ? 1 : 0, g->a15f ? 1 : 0);
        d.pad = 0;
        d.c = g->coef;
        slabs = slabs || g->slab;
    }
    // Columns of a grid's tiles, and the rows it computes (all of them, or a
    // slab's own rows between its ghosts).
    auto strips = [&](size_t k, int per) {  // per: steps of a pass
        const lbm_grid *g = b->grids[k];
        const int w = per > 1 ? fused_cols(g->storage, per) : 32 * batch_vec(b, g);
        return (g->nx + w - 1) / w;
    };
    auto computed_rows = [&](size_t k) { return b->grids[k]->ny - 2 * b->grids[k]->slab; };
    // Appends the tiles of grid k at a tile height.
    auto add_tiles = [&](size_t k, int rows, int per) {
        lbm_grid *g = b->grids[k];
        GridDesc &d = gd[k];
        w.per[k] = per;
        const int w = per > 1 ? fused_cols(g->storage, per) : 32 * batch_vec(b, g);
        const int ylo = g->slab, yhi = g->ny - g->slab, nyc = yhi - ylo;
        d.tile0 = (int)tiles.size();
        d.nstrips = strips(k, per);
        d.nsegs = (nyc + rows - 1) / rows;
        d.ntile = d.nstrips * d.nsegs;
        // A pass reads two rows and columns per step beyond its tile: the next
        // segment or strip over suffices unless one of them is smaller (the
        // last one of a grid can be).
        const int reach = 2 * per;
        const int last_rows = nyc - (d.nsegs - 1) * rows;
        const int last_cols = g->nx - (d.nstrips - 1) * w;
        d.dseg = (rows >= reach && last_rows >= reach) ? 1 : 2;
        d.dstrip = last_cols >= reach ? 1 : 2;
        // Neighbouring segments walk in opposite directions, so the rows they
        // share are read by both at about the same time (from L2 the second time).
        for (int y0 = ylo, seg = 0; y0 < yhi; y0 += rows, ++seg)
            for (int x0 = 0; x0 < g->nx; x0 += w)
                tiles.push_back(Tile{(int)k, x0, y0, std::min(yhi, y0 + rows),
                                     (seg & 1) ? -1 : 1});
    };
    // The same for passes of `per` steps in lockstep, where a last narrow strip's
    // segments share warps.
    auto add_fused_tiles = [&](size_t k, int rows, int per) {
        const lbm_grid *g = b->grids[k];
        w.per[k] = per;
        const FusedStrips s = fused_strips(g->storage, per, g->nx);
        const int w = fused_cols(g->storage, per), step = s.pieces ? s.pieces : 1;
        for (int y0 = 0, seg = 0; y0 < g->ny; y0 += rows, ++seg) {
            const int dir = (seg & 1) ? -1 : 1;
            for (int j = 0; j < s.full; ++j)
                tiles.push_back(Tile{(int)k, j * w, y0, std::min(g->ny, y0 + rows), dir});
            if (!s.pieces || seg % step) continue;
            const int y1 = (int)std::min<long long>(g->ny, y0 + (long long)step * rows);
            Tile t{(int)k, s.full * w, y0, y1, (seg / step & 1) ? -1 : 1};
            t.lanes = s.lanes;
            t.rows = std::min(rows, y1 - y0);
            tiles.push_back(t);
        }
    };
    if (b->schedule == LBM_SCHEDULE_FLOW) {
        // One launch over every grid, tiles grid by grid in their order, by the
        // kernel for the grids' kinds.  Slabs take single steps: their ghost
        // rows serve one.
        std::vector<int> kinds;
        for (const GridDesc &d : gd) kinds.push_back(d.kind);
        FlowChoice fc = flow_kernel_for(kinds, b->walk16, !slabs && !singles_only);
        lbm_batch::Group gr;
        long long warps = 0;
        auto take = [&]() -> int {
            gr.fkernel = fc.fn;
            gr.smem = fc.smem;
            gr.fused = fc.fused;
            int rc = resident_blocks(b, (const void *)fc.fn, fc.smem, &gr.max_blocks_per_sm);
            if (rc != LBM_OK) return rc;
            const int per = b->blocks_per_sm > 0 ? std::min(b->blocks_per_sm, gr.max_blocks_per_sm)
                                                 : gr.max_blocks_per_sm;
            warps = (long long)per * b->sms * kBatchWarps;
            return LBM_OK;
        };
        int rc = take();
        if (rc != LBM_OK) return rc;
        // A grid's pass takes at least one tile walk, so a grid with fewer tiles than
        // its share of the resident warps (the warps split evenly between the grids)
        // uses shorter tiles: a quarter as tall in single steps; on the fused walk as
        // tall as seven tenths of its share of warps ask for, from its reach (so that
        // a tile waits for its neighbours only) up to a height that depends on the
        // whole batch: 48 rows if that still leaves two and a half tiles a warp, else
        // 32 or 24.  Measured: 20 grids of 128^2 to 2048^2 with 1e9 updates between
        // them 8.9, 8.7, 8.4 ms at 48, 32, 24 rows; nine 2048^2 FP32 grids 174k, 168k,
        // 161k MLUPS; 512 uneven grids 138k, 131k, 120k.  Where one wave holds all tiles
        // anyway, up to the whole share: nine 512^2 FP32 grids 118k -> 134k, 32 FP16 ones
        // of 200 x 300 109k -> 131k.
        int tenths = 7;  // of a grid's share of the warps
        auto flow_rows = [&](size_t k, int tallest) {
            const long long share = std::max<long long>(1, tenths * warps / (10 * (long long)ng));
            const long long r = ((long long)strips(k, 2) * computed_rows(k) + share - 1) / share;
            return std::max(4, (int)std::min<long long>(tallest, r));
        };
        int tallest = 48;
        auto total = [&] {
            long long n = 0;
            for (size_t k = 0; k < ng; ++k) {
                const int r = flow_rows(k, tallest);
                n += (long long)strips(k, 2) * ((computed_rows(k) + r - 1) / r);
            }
            return n;
        };
        if (fc.fused && b->fit_rows) {
            for (int h : {48, 32, 24}) {
                tallest = h;
                if (2 * total() >= 5 * warps) break;
            }
            while (tenths < 10 && total() < warps) {
                ++tenths;
                if (total() > warps) {
                    --tenths;
                    break;
                }
            }
        }
        auto fused_height = [&](size_t k) {
            return b->fit_rows ? flow_rows(k, tallest) : std::max(4, b->rows);
        };
        // A 16-bit batch whose strips of 240 columns are badly filled, or whose tiles
        // come out short, is faster in single steps of 256-column strips.  Estimates of
        // a step in microseconds, as for a single grid's passes.  Measured, single /
        // fused, k MLUPS: FP16 64 grids of 256^2 140 / 108, nine of 512^2 147 / 113, 64
        // of 512^2 166 / 165, 32 of 200 x 300 119 / 131, 128 of 128^2 74 / 93, nine of
        // 2048^2 160 / 238; with stochastic rounding 64 of 256^2 109 / 93 (BF16 108 /
        // 102), nine of 512^2 107 / 98 (BF16 106 / 111), 32 of 200 x 300 88 / 113.
        //
        // FP32 and 16-bit grids together take single steps where the batch is small and
        // the fused walk's strips have a fifth more columns than those of single
        // steps (k MLUPS, single / fused: 8 grids of 256^2 42.7 / 34.4, 16 60 / 53, four
        // of 512^2 64 / 59, nine 71 / 90, 32 of 128^2 35.3 / 33.7, ten of 200^2 33 / 35,
        // eight of 384^2 51 / 64).
        const int storage = b->grids[0]->storage;
        bool one_kind = true;
        for (int kd : kinds) one_kind = one_kind && kd == kinds[0];
        bool singles = false;
        if (fc.fused && !one_kind) {
            double sites = 0, fused = 0, single = 0;
            for (size_t k = 0; k < ng; ++k) {
                const lbm_grid *g = b->grids[k];
                sites += (double)g->nx * computed_rows(k);
                fused += (double)strips(k, 2) * fused_cols(g->storage, 2) * computed_rows(k);
                single += 32.0 * strips(k, 1) * batch_vec(b, g) * computed_rows(k);
            }
            singles = sites < 1.1e6 && fused > 1.2 * single;
        }
        if (fc.fused && one_kind) {
            const bool rnd = b->grids[0]->rounding != 0, field = b->grids[0]->a15f != nullptr;
            double work = 0, pass = 0, sites = 0, single = rnd ? 5.0 : 4.0;
            double strip_sites = 0, extra = 0;
            for (size_t k = 0; k < ng; ++k) {
                const int r = fused_height(k), ny = computed_rows(k), nx = b->grids[k]->nx;
                const int segs = (ny + r - 1) / r, over = fused_overhead(2);
                work += (double)strips(k, 2) * (ny + over * segs);
                pass = std::max(pass, (double)std::min(r, ny) + over);
                const double lanes = 256.0 * strips(k, 1) / nx;
                sites += (double)nx * ny;
                single += 1e-6 * nx * ny * ((rnd ? 6.5 : 5.5) + 5.3 * (lanes - 1));
                strip_sites += 128.0 * strips(k, 1) * ny;
                extra += (double)(strips(k, 2) - strips(k, 1)) * ny;
            }
            const double passes = std::max(pass, work / warps);
            if (storage != ST_F32) {
                const double row_us = rnd ? (storage == ST_F16 ? 2.58 : 2.41) : 2.2;
                singles = single < 0.5 * row_us * passes + 0.25e-6 * sites;
            } else if (extra > 0) {
                // FP32: strips of 120 columns where single steps have fewer of 128, which
                // shows while the tiles are one wave (single / fused, us a step: 64 grids
                // of 124 x 128 13.3 / 15.5, 128 of 124 x 64 13.9 / 16.1, 32 of 128 x 256
                // 12.5 / 13.3, 16 of 128 x 512 12.6 / 13.0, nine of 128 x 4096 61 / 48, 64
                // of 248 x 128 28 / 20; with a c2 field 64 of 124 x 128 14.8 / 16.3).
                singles = std::max((field ? 9.9 : 8.5) + 4.3e-6 * strip_sites + 0.008 * ng,
                                   (field ? 14.2e-6 : 12.9e-6) * strip_sites) <
                          (field ? 0.73 : 0.715) * passes + 0.25e-6 * sites + 0.006 * ng;
            }
        }
        if (singles) {
            fc = flow_kernel_for(kinds, b->walk16, false);
            rc = take();
            if (rc != LBM_OK) return rc;
        }
        const int per_pass = fc.fused ? 2 : 1;
        for (size_t k = 0; k < ng; ++k) {
            int rows = b->rows;
            if (fc.fused) {
                rows = fused_height(k);
            } else {
                const long long tall =
                    (long long)strips(k, 1) * ((computed_rows(k) + rows - 1) / rows);
                if (tall * (long long)ng < warps) rows = std::max(1, rows / 4);
            }
            add_tiles(k, rows, per_pass);
            if (k == 0) gr.rows = rows;
        }
        gr.count = (int)tiles.size();
        w.groups.push_back(gr);
        if (tiles.size() > b->prog_cap) {
            int *prog = nullptr;
            BCK(cudaMalloc(&prog, sizeof(int) * tiles.size()));
            cudaFree(b->d_prog);
            b->d_prog = prog;
            b->prog_cap = tiles.size();
            drop_graphs(b);  // (both lists' launches use it)
        }
        if (!b->d_ctl)
            BCK(cudaMalloc(&b->d_ctl, sizeof(unsigned long long) * kFlowCtlWords * ng));
        return upload_worklist(b, w, gd, tiles);
    }
    // Lockstep, default configuration, single-step walks: every warp walks its
    // tiles one after another within a step, so a batch with fewer tiles than
    // about the resident warps (16 per SM in the specialised kernels) spends
    // each step on a whole walk with warps idle.  Such a batch gets shorter
    // tiles, down to 2 rows, as many as one wave holds.  Batches of at least
    // 3/4 of a wave of tiles keep the configured height.
    int lock_rows = b->rows;
    if (b->fit_rows) {
        const int bps = b->blocks_per_sm > 0 ? b->blocks_per_sm : 4;
        const long long wave = (long long)bps * b->sms * kBatchWarps;
        auto tiles_at = [&](int r) {
            long long t = 0;
            for (size_t k = 0; k < ng; ++k)
                t += (long long)strips(k, 1) * ((computed_rows(k) + r - 1) / r);
            return t;
        };
        if (4 * tiles_at(lock_rows) < 3 * wave)
            while (lock_rows > 2 && tiles_at(lock_rows - 1) <= wave) --lock_rows;
    }
    // Kind groups.  A kind with a specialised kernel runs in its own launch
    // when its grids move at least kOwnLaunchBytes per step (about 10 us of
    // HBM time, so the launch's fixed costs and its barrier stay small); all
    // other tiles share one launch of the general kernel, where small grids of
    // any kind overlap.  A batch of one kind is one group.
    constexpr double kOwnLaunchBytes = 64.0 * 1024 * 1024;
    std::vector<double> bytes(kKindCodes, 0.0);
    std::vector<std::vector<size_t>> of_kind(kKindCodes);
    int kinds_present = 0;
    for (size_t k = 0; k < ng; ++k) {
        const lbm_grid *g = b->grids[k];
        bytes[gd[k].kind] += (double)g->nx * computed_rows(k) *
                             ((g->storage == ST_F32 ? 72.0 : 36.0) + (g->a15f ? 4.0 : 0.0));
        kinds_present += of_kind[gd[k].kind].empty();
        of_kind[gd[k].kind].push_back(k);
    }
    std::vector<Tile> ordered;
    // A group of one 8-site 16-bit kind (automatic walk) pairs the tiles of
    // its grids at most kSplitCols wide: consecutive segments share one warp,
    // a half-warp each (the split walk), where a single walk leaves half of
    // the lanes or more idle.  An odd one out stays single.  The kernel
    // instance with the split walk runs the whole-warp walk a few per cent
    // slower (its register allocation), and pairing the narrow last strip of
    // a wider grid measured no faster, so a group pairs only whole narrow
    // grids, and only when their tiles are at least kSplitMinShare of its
    // tiles.
    auto splits = [&](int kd) {
        if (!kind_splits(kd) || b->walk16 != LBM_WALK16_AUTO) return false;
        long long n_all = 0, n_narrow = 0;
        for (size_t k : of_kind[kd]) {
            const long long n =
                (long long)strips(k, 1) * ((computed_rows(k) + lock_rows - 1) / lock_rows);
            n_all += n;
            if (gd[k].nx <= kSplitCols) n_narrow += n;
        }
        return n_narrow > 0 && (double)n_narrow >= kSplitMinShare * (double)n_all;
    };
    // The fused walk serves every group of one kind that
    // has it, but for the split walk's groups, slabs, and 16-bit walks the
    // caller chose.
    auto fuses = [&](int kd) {
        if (singles_only || !fused_kernel_for(kd, 2).fn || splits(kd)) return false;
        for (size_t k : of_kind[kd])
            if (b->grids[k]->slab ||
                (b->grids[k]->storage != ST_F32 && b->walk16 != LBM_WALK16_AUTO))
                return false;
        return true;
    };
    // The end of each pass: the warps that take the last tiles set its length,
    // and the others wait at the barrier.  A group of more than two waves of
    // tiles splits its last wave's tiles in two (8 rows each at the default
    // height), halving that tail for a few more pulled rows per split tile.
    // Measured with single steps: the nine 2048^2 FP16-delta grids 168.1k ->
    // 170.2k MLUPS (stochastic rounding 165.0k -> 168.0k), the 512-grid batch
    // FP16-delta 158.6k -> 159.4k, FP32 sweep 93.4k -> 93.8k; quarters, or
    // halves over the last two waves, gained less.
    auto split_tail = [&](size_t begin, long long wave) {
        if ((long long)(ordered.size() - begin) <= 2 * wave) return;
        std::vector<Tile> tail(ordered.end() - wave, ordered.end());
        ordered.resize(ordered.size() - wave);
        for (const Tile &t : tail) {
            if (t.y1b > t.y0b || t.lanes || t.y1 - t.y0 < 2) {
                ordered.push_back(t);
                continue;
            }
            const int mid = t.y0 + (t.y1 - t.y0) / 2;
            ordered.push_back(Tile{t.grid, t.x0, t.y0, mid, 1});
            ordered.push_back(Tile{t.grid, t.x0, mid, t.y1, -1});
        }
    };
    auto add_group = [&](const std::vector<int> &kinds_in) -> int {
        lbm_batch::Group gr;
        gr.begin = (int)ordered.size();
        tiles.clear();
        bool fused = kinds_in.size() == 1 && fuses(kinds_in[0]);
        int per = 2;
        long long warps = 1;
        if (fused) {
            const std::vector<size_t> &members = of_kind[kinds_in[0]];
            const int storage = b->grids[members[0]]->storage;
            const bool field = b->grids[members[0]]->a15f != nullptr;
            double best = 1e300;
            // (with a c2 field three steps gain nothing here: 22.5 ms against 22.4)
            for (int steps = 2; steps <= (field ? 2 : fused_most_steps(storage)); ++steps) {
                const FusedChoice fc = fused_kernel_for(kinds_in[0], steps);
                int bps = 0;
                int rc = resident_blocks(b, (const void *)fc.fn, fc.smem, &bps);
                if (rc != LBM_OK) return rc;
                const long long w =
                    (long long)(b->blocks_per_sm > 0 ? std::min(b->blocks_per_sm, bps) : bps) *
                    b->sms * kBatchWarps;
                std::vector<std::pair<FusedStrips, int>> shape;
                for (size_t k : members)
                    shape.push_back({fused_strips(storage, steps, b->grids[k]->nx),
                                     computed_rows(k)});
                double cost = 0;
                const int rows = fused_rows(shape, w, fused_overhead(steps),
                                            fused_most_rows(storage, steps),
                                            b->fit_rows ? 0 : b->rows, &cost);
                // A row step of three steps takes about 1.4 times as long as one of
                // two here, in a launch per pass 1.22 times (nine 2048^2 grids, three
                // steps and 296 rows 20.2 ms for 100, two and 56 rows 21.4).
                cost /= steps == 3 ? 3 / 1.42 : 2.0;
                if (cost >= best) continue;
                best = cost;
                per = steps;
                gr.kernel = fc.fn;
                gr.smem = fc.smem;
                gr.max_blocks_per_sm = bps;
                gr.rows = rows;
                warps = w;
            }
            // FP32 strips are 120 columns here and 128 in single steps, so widths of 121 to
            // 128 (or 241 to 256, less so) have one more; a batch of less than a wave of
            // tiles then is the faster in single steps.  Estimates of a step as above.
            // Single / fused, us a step: 64 grids of 124 x 128 14.6 / 15.8, 128 of 124 x 64
            // 14.6 / 16.5, 256 of 124 x 32 14.6 / 16.5, 16 of 124 x 512 14.6 / 15.2, 64 of
            // 124 x 256 27.1 / 26.1, 64 of 116 x 128 14.6 / 10.0, 64 of 248 x 128 27 / 20;
            // with a c2 field 128 of 124 x 64 16.3 / 16.7.
            if (storage == ST_F32 && b->fit_rows && lock_rows < b->rows) {
                double strip_sites = 0, extra = 0;
                for (size_t k : members) {
                    strip_sites += 128.0 * strips(k, 1) * computed_rows(k);
                    extra += (double)(strips(k, 2) - strips(k, 1)) * computed_rows(k);
                }
                const double single = std::max((field ? 7.3 : 6.5) + (field ? 2.2 : 2.05) * lock_rows,
                                               13.3e-6 * strip_sites);
                if (extra > 0 && single < (field ? 1.46 : 1.43) * best + 1.5) fused = false;
            }
        }
        if (fused) {
            gr.fused = true;
            for (size_t k : of_kind[kinds_in[0]]) add_fused_tiles(k, gr.rows, per);
            ordered.insert(ordered.end(), tiles.begin(), tiles.end());
            split_tail(gr.begin, warps);
            gr.count = (int)ordered.size() - gr.begin;
            w.groups.push_back(gr);
            return LBM_OK;
        }
        gr.smem = 0;
        for (int kd : kinds_in)
            for (size_t k : of_kind[kd]) add_tiles(k, lock_rows, 1);
        // (grids in the caller's order, whatever their kinds)
        std::stable_sort(tiles.begin(), tiles.end(),
                         [](const Tile &x, const Tile &y) { return x.grid < y.grid; });
        const bool split = kinds_in.size() == 1 && splits(kinds_in[0]);
        const int paired0 = w.paired;
        std::vector<int> pending(ng, -1);
        for (const Tile &t : tiles) {
            if (split && gd[t.grid].nx <= kSplitCols) {
                int &p = pending[t.grid];
                if (p >= 0) {
                    Tile &a = ordered[p];
                    a.y0b = t.y0;
                    a.y1b = t.y1;
                    a.dirb = t.dir;
                    p = -1;
                    ++w.paired;
                    continue;
                }
                p = (int)ordered.size();
            }
            ordered.push_back(t);
        }
        const int bps = b->blocks_per_sm > 0 ? b->blocks_per_sm : 4;
        split_tail(gr.begin, (long long)bps * b->sms * kBatchWarps);
        gr.rows = lock_rows;
        gr.count = (int)ordered.size() - gr.begin;
        gr.kernel = kernel_for(kinds_in, b->walk16, w.paired > paired0);
        int rc = resident_blocks(b, (const void *)gr.kernel, 0, &gr.max_blocks_per_sm);
        if (rc != LBM_OK) return rc;
        w.groups.push_back(gr);
        return LBM_OK;
    };
    std::vector<int> rest;
    for (int kd = 0; kd < kKindCodes; ++kd) {
        if (of_kind[kd].empty()) continue;
        BatchKernel kk = kernel_for({kd}, b->walk16);
        if (kk != (BatchKernel)k_batch && (kinds_present == 1 || bytes[kd] >= kOwnLaunchBytes)) {
            int rc = add_group({kd});
            if (rc != LBM_OK) return rc;
        } else {
            rest.push_back(kd);
        }
    }
    if (!rest.empty()) {
        int rc = add_group(rest);
        if (rc != LBM_OK) return rc;
    }
    return upload_worklist(b, w, gd, ordered);
}

// (Re)builds the batch's work-list after a change of its settings; the list for calls of
// one step follows when one needs it.
static int build_worklist(lbm_batch *b) {
    b->list[1].built = false;
    return build_list(b, b->list[0], false);
}

extern "C" int lbm_batch_destroy(lbm_batch_t b) {
    if (!b) return LBM_OK;
    if (b->stream || b->d_limit) cudaStreamSynchronize(b->stream);
    drop_graphs(b);
    for (lbm_batch::List &w : b->list) {
        cudaFree(w.d_grids);
        cudaFree(w.d_tiles);
    }
    cudaFree(b->d_limit);
    cudaFree(b->d_parity);
    cudaFree(b->d_t0);
    cudaFree(b->d_bar);
    cudaFree(b->d_status);
    cudaFree(b->d_ctl);
    cudaFree(b->d_prog);
    cudaFree(b->d_nwork);
    if (b->h_nwork) cudaFreeHost(b->h_nwork);
    if (b->h_limit) cudaFreeHost(b->h_limit);
    if (b->h_parity) cudaFreeHost(b->h_parity);
    if (b->h_t0) cudaFreeHost(b->h_t0);
    if (b->h_status) cudaFreeHost(b->h_status);
    if (b->copied) cudaEventDestroy(b->copied);
    for (cudaEvent_t ev : b->xev) cudaEventDestroy(ev);
    if (b->done) cudaEventDestroy(b->done);
    delete b;
    return LBM_OK;
}

extern "C" int lbm_batch_create(const lbm_t *grids, int n, lbm_batch_t *out) {
    if (!out || !grids || n < 1) return bfail(LBM_EINVAL, "lbm_batch_create: bad argument");
    *out = nullptr;
    for (int k = 0; k < n; ++k) {
        if (!grids[k]) return bfail(LBM_EINVAL, "lbm_batch_create: NULL grid");
        if (grids[k]->drive)
            return bfail(LBM_EINVAL, "lbm_batch_create: driven grids are not batched");
        if (grids[k]->grad != LBM_GRAD_CENTRAL)
            return bfail(LBM_EINVAL, "lbm_batch_create: the batch kernels use the central "
                                     "difference (lbm_set_gradient)");
    }
    lbm_batch *b = new (std::nothrow) lbm_batch();
    if (!b) return bfail(LBM_ENOMEM, "lbm_batch_create: host allocation failed");
    b->grids.assign(grids, grids + n);
    b->stream = grids[0]->stream;
    b->device = grids[0]->device;
    for (int k = 0; k < n; ++k)
        if (grids[k]->device != b->device) {
            delete b;
            return bfail(LBM_EINVAL, "lbm_batch_create: grids on different devices");
        }
    // One attribute (a full cudaGetDeviceProperties is slow, and servers
    // re-create batches often).
    cudaError_t e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_limit, sizeof(long long) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_parity, sizeof(int) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_t0, sizeof(uint32_t) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_bar, sizeof(unsigned) * kBarWords);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_limit, sizeof(long long) * n);
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_parity, sizeof(int) * n);
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_t0, sizeof(uint32_t) * n);
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_nwork, sizeof(int));
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_nwork, sizeof(int));
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->copied, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int));
    if (e != cudaSuccess) {
        int rc = bcuda(e, "lbm_batch_create");
        lbm_batch_destroy(b);
        return rc;
    }
    int rc = build_worklist(b);
    if (rc != LBM_OK) {
        lbm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return LBM_OK;
}

static int grid_blocks(const lbm_batch *b, const lbm_batch::Group &g) {
    int per = b->blocks_per_sm > 0 ? std::min(b->blocks_per_sm, g.max_blocks_per_sm)
                                   : g.max_blocks_per_sm;
    return per * b->sms;
}

// Queues: copy per-call arrays, reset barrier and status, cooperative launch.
static cudaError_t enqueue(lbm_batch *b, lbm_batch::List &w, long long n, cudaStream_t st) {
    int ng = (int)b->grids.size();
    cudaError_t e = cudaMemcpyAsync(b->d_limit, b->h_limit, sizeof(long long) * ng,
                                    cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_parity, b->h_parity, sizeof(int) * ng, cudaMemcpyHostToDevice,
                            st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_t0, b->h_t0, sizeof(uint32_t) * ng, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_status, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const GridDesc *grids = w.d_grids;
    const long long *lim = b->d_limit;
    const int *par = b->d_parity;
    const uint32_t *t0 = b->d_t0;
    unsigned *bar = b->d_bar;
    int *status = b->d_status;
    unsigned long long to = b->timeout_ns;
    if (b->schedule == LBM_SCHEDULE_FLOW) {
        e = cudaMemcpyAsync(b->d_nwork, b->h_nwork, sizeof(int), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(b->d_ctl, 0,
                                sizeof(unsigned long long) * kFlowCtlWords * ng, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->d_prog, 0, sizeof(int) * w.ntiles, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->d_bar, 0, sizeof(unsigned) * kBarWords, st);
        if (e != cudaSuccess) return e;
        const lbm_batch::Group &gr = w.groups[0];
        gr.fkernel<<<grid_blocks(b, gr), 32 * kBatchWarps, gr.smem, st>>>(
            grids, ng, w.d_tiles, lim, par, t0, b->d_ctl, b->d_prog, bar, b->d_nwork, status,
            to);
        return cudaGetLastError();
    }
    // The groups hold disjoint grids: each launch advances its grids by all n
    // steps.  Barrier words and tile counters start at zero for every launch.
    for (const lbm_batch::Group &gr : w.groups) {
        e = cudaMemsetAsync(b->d_bar, 0, sizeof(unsigned) * kBarWords, st);
        if (e != cudaSuccess) return e;
        const Tile *tiles = w.d_tiles + gr.begin;
        int ntiles = gr.count;
        void *args[] = {(void *)&grids, (void *)&tiles, (void *)&ntiles, (void *)&lim,
                        (void *)&par,   (void *)&t0,    (void *)&n,      (void *)&bar,
                        (void *)&status, (void *)&to};
        e = cudaLaunchCooperativeKernel((const void *)gr.kernel, dim3(grid_blocks(b, gr)),
                                        dim3(32 * kBatchWarps), args, gr.smem, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static int run_batch(lbm_batch *b, lbm_batch::List &w, long long n, const long long *limits,
                     bool advance) {
    int ng = (int)b->grids.size();
    // The previous call's copies must have read the pinned arrays first.
    BCK(cudaEventSynchronize(b->copied));
    int nwork = 0;
    for (int k = 0; k < ng; ++k) {
        long long lim = limits ? std::max(0LL, std::min(n, limits[k])) : n;
        b->h_limit[k] = lim;
        b->h_parity[k] = b->grids[k]->cur;
        b->h_t0[k] = (uint32_t)b->grids[k]->t;
        nwork += lim > 0;
    }
    *b->h_nwork = nwork;
    // Work already queued on the members' own streams (an lbm_init, a step
    // call) runs before the batch's launches.
    int nxs = 0;
    for (const lbm_grid *g : b->grids) {
        cudaStream_t s = g->stream;
        if (s == b->stream || std::find(b->xs.begin(), b->xs.begin() + nxs, s) != b->xs.begin() + nxs)
            continue;
        if (nxs == (int)b->xs.size()) {
            cudaEvent_t ev = nullptr;
            BCK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
            b->xev.push_back(ev);
            b->xs.push_back(s);
        }
        b->xs[nxs] = s;
        BCK(cudaEventRecord(b->xev[nxs], s));
        BCK(cudaStreamWaitEvent(b->stream, b->xev[nxs], 0));
        ++nxs;
    }
    cudaError_t e = cudaSuccess;
    const bool want_graph = b->launch_mode == LBM_LAUNCH_GRAPH ||
                            (b->launch_mode == LBM_LAUNCH_AUTO && !b->capture_failed);
    bool graphed = false;
    if (want_graph) {
        if (w.graph_n != n) {
            drop_graph(w);
            cudaStream_t cs;
            BCK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
            cudaGraph_t g = nullptr;
            e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                cudaError_t e1 = enqueue(b, w, n, cs);
                cudaError_t e2 = cudaStreamEndCapture(cs, &g);
                e = e1 != cudaSuccess ? e1 : e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&w.graph, g, 0);
            if (g) cudaGraphDestroy(g);
            cudaStreamDestroy(cs);
            if (e != cudaSuccess) {
                cudaGetLastError();
                drop_graph(w);
                if (b->launch_mode == LBM_LAUNCH_GRAPH)
                    return bcuda(e, "lbm_batch_step: capturing the persistent launch in a CUDA graph");
                // AUTO: recorded (lbm_batch_get_launch) and never retried.
                b->capture_failed = true;
            } else {
                w.graph_n = n;
            }
        }
        if (w.graph) {
            e = cudaGraphLaunch(w.graph, b->stream);
            graphed = true;
        }
    }
    if (!graphed) e = enqueue(b, w, n, b->stream);
    if (e != cudaSuccess) return bcuda(e, "lbm_batch_step launch");
    b->last_launch = graphed ? LBM_LAUNCH_GRAPH : LBM_LAUNCH_DIRECT;
    BCK(cudaEventRecord(b->copied, b->stream));
    if (nxs) {
        // Later work on those streams (lbm_moments, lbm_destroy, a step)
        // waits for the batch's.
        BCK(cudaEventRecord(b->done, b->stream));
        for (int k = 0; k < nxs; ++k) BCK(cudaStreamWaitEvent(b->xs[k], b->done, 0));
    }
    if (advance) {
        for (int k = 0; k < ng; ++k) {
            long long s = b->h_limit[k];
            b->grids[k]->t += s;
            if (passes_of(s, w.per[k]) & 1) b->grids[k]->cur ^= 1;
        }
    }
    return LBM_OK;
}

// Builds a list that is not the one of the batch's settings and grids.
static int ready(lbm_batch *b, lbm_batch::List &w, bool singles_only) {
    bool stale = !w.built;
    for (size_t k = 0; k < b->grids.size() && !stale; ++k) {
        const lbm_grid *g = b->grids[k];
        stale = g->a15f != w.built_a15f[k] || g->rounding != w.built_rounding[k];
    }
    if (!stale) return LBM_OK;
    BCK(cudaStreamSynchronize(b->stream));
    return build_list(b, w, singles_only);
}

extern "C" int lbm_batch_step(lbm_batch_t b, long long n, const long long *limits) {
    if (!b || n < 0) return bfail(LBM_EINVAL, "lbm_batch_step: bad argument");
    if (b->schedule == LBM_SCHEDULE_FLOW && n > 0x7fffffffLL)
        return bfail(LBM_EINVAL, "lbm_batch_step: flow schedule takes at most 2^31 - 1 steps a call");
    if (n == 0) return LBM_OK;
    for (const lbm_grid *g : b->grids) {
        if (g->drive) return bfail(LBM_EINVAL, "lbm_batch_step: a grid has a drive");
        if (g->grad != LBM_GRAD_CENTRAL)
            return bfail(LBM_EINVAL, "lbm_batch_step: a grid uses the forward difference");
    }
    int rc = ready(b, b->list[0], false);
    if (rc != LBM_OK) return rc;
    const std::vector<int> &per = b->list[0].per;
    const bool single = n == 1 && *std::max_element(per.begin(), per.end()) > 1;
    if (single && (rc = ready(b, b->list[1], true)) != LBM_OK) return rc;
    return run_batch(b, b->list[single ? 1 : 0], n, limits, true);
}

cudaError_t batch_queue_status(lbm_batch *b, cudaStream_t st) {
    return cudaMemcpyAsync(b->h_status, b->d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
}

int batch_status(const lbm_batch *b) { return *b->h_status; }

extern "C" int lbm_batch_sync(lbm_batch_t b) {
    if (!b) return bfail(LBM_EINVAL, "lbm_batch_sync: NULL batch");
    BCK(cudaMemcpyAsync(b->h_status, b->d_status, sizeof(int), cudaMemcpyDeviceToHost,
                        b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    if (*b->h_status != 0)
        return bfail(*b->h_status, "lbm_batch_sync: a barrier wait in the batch kernel ran out");
    return LBM_OK;
}

extern "C" int lbm_batch_set_config(lbm_batch_t b, int rows, int blocks_per_sm) {
    if (!b || rows < 1 || rows > 4096 || blocks_per_sm < 0)
        return bfail(LBM_EINVAL, "lbm_batch_set_config: bad argument");
    BCK(cudaStreamSynchronize(b->stream));
    b->blocks_per_sm = blocks_per_sm;
    if (rows != b->rows || b->fit_rows || !b->list[0].built) {
        b->rows = rows;
        b->fit_rows = false;
        return build_worklist(b);
    }
    drop_graphs(b);
    return LBM_OK;
}

extern "C" int lbm_batch_set_walk16(lbm_batch_t b, int walk) {
    if (!b || walk < LBM_WALK16_AUTO || walk > LBM_WALK16_V4_PF2)
        return bfail(LBM_EINVAL, "lbm_batch_set_walk16: unknown walk");
    BCK(cudaStreamSynchronize(b->stream));
    if (walk == b->walk16 && b->list[0].built) return LBM_OK;
    b->walk16 = walk;
    return build_worklist(b);
}

extern "C" int lbm_batch_get_walk16(lbm_batch_t b, int *walk) {
    if (!b || !walk) return bfail(LBM_EINVAL, "lbm_batch_get_walk16: bad argument");
    *walk = b->walk16;
    return LBM_OK;
}

extern "C" int lbm_batch_get_groups(lbm_batch_t b, int *groups) {
    if (!b || !groups) return bfail(LBM_EINVAL, "lbm_batch_get_groups: bad argument");
    *groups = (int)b->list[0].groups.size();
    return LBM_OK;
}

extern "C" int lbm_batch_set_timeout_us(lbm_batch_t b, long long us) {
    if (!b || us < 1) return bfail(LBM_EINVAL, "lbm_batch_set_timeout_us: bad argument");
    b->timeout_ns = (unsigned long long)us * 1000ULL;
    drop_graphs(b);
    return LBM_OK;
}

// A configuration the tuner tries: a tile height (0: the heights the work-list
// fits by itself) and a 16-bit walk.
struct BatchTry {
    int rows, walk;
};

static int apply_try(lbm_batch *b, const BatchTry &t) {
    int rc = lbm_batch_set_walk16(b, t.walk);
    if (rc != LBM_OK) return rc;
    if (t.rows > 0) return lbm_batch_set_config(b, t.rows, 0);
    b->rows = 16;
    b->fit_rows = true;
    b->blocks_per_sm = 0;
    return build_worklist(b);
}

// Milliseconds per 1e9 lattice updates of dry passes (the state is not
// advanced: every grid writes its other buffer) under the work-list as built,
// at its full occupancy.  A pass is one step, or several for a grid on the
// fused walk; it does the same work as a pass inside a longer launch (the barriers
// cost microseconds per millisecond pass).
static int time_passes(lbm_batch *b, cudaEvent_t e0, cudaEvent_t e1, double *cost) {
    std::vector<long long> limits;
    long long most = 1;
    double updates = 0;
    for (size_t k = 0; k < b->grids.size(); ++k) {
        const lbm_grid *g = b->grids[k];
        limits.push_back(b->list[0].per[k]);
        most = std::max(most, limits.back());
        updates += (double)limits.back() * g->nx * (g->ny - 2 * g->slab);
    }
    int rc = run_batch(b, b->list[0], most, limits.data(), false);  // warm-up (and graph build)
    if (rc != LBM_OK) return rc;
    BCK(cudaEventRecord(e0, b->stream));
    for (int k = 0; k < 4 && rc == LBM_OK; ++k) rc = run_batch(b, b->list[0], most, limits.data(), false);
    if (rc != LBM_OK) return rc;
    BCK(cudaEventRecord(e1, b->stream));
    BCK(cudaEventSynchronize(e1));
    float ms = 0.f;
    BCK(cudaEventElapsedTime(&ms, e0, e1));
    *cost = ms / 4 / updates * 1e9;
    return LBM_OK;
}

// Times several tile heights, when the batch holds 16-bit grids the 16-bit
// walks, and with groups on the fused walk the heights the work-list fits by
// itself; leaves the fastest in *best.
static int tune_candidates(lbm_batch *b, cudaEvent_t e0, cudaEvent_t e1, BatchTry *best) {
    double least = 1e300;
    std::vector<std::vector<BatchKernel>> seen;
    for (int walk = LBM_WALK16_AUTO; walk <= LBM_WALK16_V4_PF2; ++walk) {
        int rc = lbm_batch_set_walk16(b, walk);
        if (rc != LBM_OK) return rc;
        std::vector<BatchKernel> ks;
        bool fused = false;
        for (const auto &gr : b->list[0].groups) {
            ks.push_back(gr.kernel);
            fused = fused || gr.fused;
        }
        if (std::find(seen.begin(), seen.end(), ks) != seen.end()) continue;  // same kernels
        seen.push_back(ks);
        for (int r : {0, 8, 12, 16, 24, 32}) {
            if (r == 0 && !fused) continue;
            double cost = 0;
            rc = apply_try(b, BatchTry{r, walk});
            if (rc == LBM_OK) rc = time_passes(b, e0, e1, &cost);
            if (rc != LBM_OK) return rc;
            if (cost < least) {
                least = cost;
                *best = BatchTry{r, walk};
            }
        }
    }
    return LBM_OK;
}

extern "C" int lbm_batch_tune(lbm_batch_t b) {
    if (!b) return bfail(LBM_EINVAL, "lbm_batch_tune: NULL batch");
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    BCK(cudaEventCreate(&e0));
    cudaError_t e = cudaEventCreate(&e1);
    if (e != cudaSuccess) {
        cudaEventDestroy(e0);
        return bcuda(e, "cudaEventCreate");
    }
    const int rows0 = b->rows, walk0 = b->walk16, bps0 = b->blocks_per_sm;
    const bool fit0 = b->fit_rows;
    BatchTry best{rows0, walk0};
    int rc = tune_candidates(b, e0, e1, &best);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc != LBM_OK) {
        // The configuration in force before the call is put back.
        lbm_batch_set_walk16(b, walk0);
        lbm_batch_set_config(b, rows0, bps0);
        if (fit0) {
            b->fit_rows = true;
            build_worklist(b);
        }
        return rc;
    }
    return apply_try(b, best);
}

extern "C" int lbm_batch_set_schedule(lbm_batch_t b, int schedule) {
    if (!b || schedule < LBM_SCHEDULE_LOCKSTEP || schedule > LBM_SCHEDULE_FLOW)
        return bfail(LBM_EINVAL, "lbm_batch_set_schedule: unknown schedule");
    BCK(cudaStreamSynchronize(b->stream));
    if (schedule == b->schedule && b->list[0].built) return LBM_OK;
    b->schedule = schedule;
    return build_worklist(b);
}

extern "C" int lbm_batch_get_schedule(lbm_batch_t b, int *schedule) {
    if (!b || !schedule) return bfail(LBM_EINVAL, "lbm_batch_get_schedule: bad argument");
    *schedule = b->schedule;
    return LBM_OK;
}

extern "C" int lbm_batch_set_launch(lbm_batch_t b, int mode) {
    if (!b || mode < LBM_LAUNCH_AUTO || mode > LBM_LAUNCH_DIRECT)
        return bfail(LBM_EINVAL, "lbm_batch_set_launch: unknown mode");
    BCK(cudaStreamSynchronize(b->stream));
    b->launch_mode = mode;
    b->capture_failed = false;
    drop_graphs(b);
    return LBM_OK;
}

extern "C" int lbm_batch_get_launch(lbm_batch_t b, int *mode, int *last, int *capture_failed) {
    if (!b) return bfail(LBM_EINVAL, "lbm_batch_get_launch: NULL batch");
    if (mode) *mode = b->launch_mode;
    if (last) *last = b->last_launch;
    if (capture_failed) *capture_failed = b->capture_failed ? 1 : 0;
    return LBM_OK;
}

extern "C" int lbm_batch_get_tiles(lbm_batch_t b, int *tiles, int *paired) {
    if (!b) return bfail(LBM_EINVAL, "lbm_batch_get_tiles: NULL batch");
    if (tiles) *tiles = b->list[0].ntiles;
    if (paired) *paired = b->list[0].paired;
    return LBM_OK;
}

extern "C" int lbm_batch_get_pass(lbm_batch_t b, int grid, int *steps) {
    if (!b || !steps || grid < 0 || grid >= (int)b->grids.size())
        return bfail(LBM_EINVAL, "lbm_batch_get_pass: bad argument");
    *steps = b->list[0].per[grid];
    return LBM_OK;
}

extern "C" int lbm_batch_get_config(lbm_batch_t b, int *rows, int *blocks_per_sm,
                                    int *specialised) {
    if (!b) return bfail(LBM_EINVAL, "lbm_batch_get_config: NULL batch");
    if (rows) *rows = b->list[0].groups.empty() ? b->rows : b->list[0].groups[0].rows;
    if (blocks_per_sm)
        *blocks_per_sm = b->list[0].groups.empty() ? 0 : grid_blocks(b, b->list[0].groups[0]) / b->sms;
    if (specialised) {
        *specialised = 1;
        for (const auto &gr : b->list[0].groups)
            if (gr.kernel == (BatchKernel)k_batch || gr.fkernel == (FlowKernel)k_flow)
                *specialised = 0;
    }
    return LBM_OK;
}
