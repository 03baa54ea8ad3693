// dfgks_decomp.cu -- one problem split into px x py rectangular blocks with halo exchange.
//
// Each block is a ghosted mesh of its own (buffers, sweeps and update as for a whole mesh); the
// ghost layers of a side it shares with another block (or of a periodic side that wraps onto
// another block) are filled by copies of that block's boundary cells instead of by a boundary
// condition.  Before every stage the ghost fill runs as two passes over all blocks, as on the
// whole mesh: (1) the ghost columns of the interior rows (physical sides by their boundary
// condition, shared sides by copying the neighbour's G boundary columns), then (2) the ghost
// rows of all columns, ghost columns included (physical sides by their boundary condition, which
// reads the columns of pass 1; shared sides by copying the neighbour's G boundary rows with its
// ghost columns).  Pass 2 carries the diagonal neighbours' cells into the corners, so no
// diagonal exchange is needed.  Every ghost cell then holds what the whole mesh's fill puts
// there, the per-cell arithmetic is the same, and a decomposed run reproduces the undivided one
// bit for bit.  All blocks share one device step state: the CFL kernels of all blocks take their
// minimum into it (the dt all-reduce of a multi-device run), and one halt flag stops them all.
//
// On one device the copies are device-to-device; the block plan (dfgks_decomp_plan) is the same
// bookkeeping a run with one block per device would use, where the copies become sends and
// receives of the same strips.
#include <cuda_runtime.h>
#include <string.h>
#include <new>
#include <vector>

#include "../../include/dfgks.h"
#include "dfgks_bodies.cuh"

using namespace dfk;

namespace {

// A block as the ghost-fill kernel sees it: its fields and, per side shared with another block, that block and
// the first cells of the two windows (halo_window)
struct HaloBlock {
    Mesh m;
    double* W[3];         // W[0], W[1], Ws
    double* A[2];
    int neighbour[4], di[4], dj[4], si[4], sj[4];
};

// One pass of the ghost fill of all blocks (grid x: block): 0 the ghost columns of the interior rows, 1 the ghost
// rows of all columns.  A pass reads no cell that it writes, so physical sides and copies go together: one launch
// instead of a launch and up to ten strided copies per block (measured with the blocks' streams, see Helpers below).
// The last pass also notes the halt flag for the updates that follow (hold, see enqueue_decomp_step).
__global__ void k_halo(const HaloBlock* __restrict__ H, int pass, int field, int alpha, const int* halt, int* hold) {
    const int halted = *(volatile const int*)halt;
    if (pass == 1 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *hold = halted;
    if (halted != 0) return;
    const HaloBlock& b = H[blockIdx.x];
    const int idx = blockIdx.y * blockDim.x + threadIdx.x;
    const Mesh& m = b.m;
    double* W = b.W[field];
    double* A = alpha >= 0 ? b.A[alpha] : nullptr;
    int i, j, g;                                          // cell and ghost layer
    if (pass == 0) {
        g = idx % (2 * G); j = idx / (2 * G);
        if (j >= m.ny) return;
        i = g < G ? g - G : m.nx + g - G;
    } else {
        i = idx % (m.nx + 2 * G) - G; g = idx / (m.nx + 2 * G);
        if (g >= 2 * G) return;
        j = g < G ? g - G : m.ny + g - G;
    }
    const int side = 2 * pass + (g < G ? 0 : 1), nb = b.neighbour[side];
    if (nb < 0) {
        if (pass == 0) ghost_x_body(m, W, A, g, j);
        else ghost_y_body(m, W, A, i, g);
        return;
    }
    const HaloBlock& a = H[nb];
    const long long d = gid(m, i, j), o = gid(a.m, b.si[side] + (i - b.di[side]), b.sj[side] + (j - b.dj[side]));
#pragma unroll
    for (int k = 0; k < 4; ++k) W[k * m.plane + d] = a.W[field][k * a.m.plane + o];
    if (A) A[d] = a.A[alpha][o];
}

struct Block {
    dfgks_block_plan plan;
    Mesh m;
    double* W[2];
    double* A[2];
    double* Ws;
    double* acc;          // dense [4][ny][nx]: S2O4 accumulator and transfer staging
    SweepBuffers B;       // x-faces' records and both flux record sets
    SweepBuffers By;      // y-faces' face-line and Gauss-point records (fused x/y sweeps)
};

long long round4(long long n) { return (n + 3) & ~3LL; }
int split(int n, int parts, int k) { return (int)(((long long)n * k) / parts); }

bool decomp_config_ok(const dfgks_config* c, int px, int py) {
    if (!c || px < 1 || py < 1 || px > 4096 || py > 4096) return false;
    if (c->nx < 1 || c->ny < 1 || c->nx > (1 << 20) || c->ny > (1 << 20)) return false;
    if (!(c->x1 > c->x0) || !(c->y1 > c->y0) || !(c->gamma > 1.0) || !(c->cfl > 0.0) || !(c->eps > 0.0)) return false;
    if (!(c->dH > 0.0 && c->dH <= 1.0) || !(c->dL >= 0.0 && c->dL <= 1.0) || !(c->C1 >= 0.0) || !(c->C2 >= 0.0)) return false;
    const int bcs[4] = {c->bc_xlo, c->bc_xhi, c->bc_ylo, c->bc_yhi};
    for (int k = 0; k < 4; ++k) if (bcs[k] < 0 || bcs[k] > 2) return false;
    if ((c->bc_xlo == 0) != (c->bc_xhi == 0) || (c->bc_ylo == 0) != (c->bc_yhi == 0)) return false;
    // a halo copy takes G boundary cells of the neighbour, and periodic or walled sides copy or
    // mirror G cells of the block itself: every block needs G cells along a split direction,
    // an unsplit direction the whole mesh's rule
    if (px > 1 && c->nx / px < G) return false;
    if (py > 1 && c->ny / py < G) return false;
    if (px == 1 && (c->bc_xlo != 1 || c->bc_xhi != 1) && c->nx < G) return false;
    if (py == 1 && (c->bc_ylo != 1 || c->bc_yhi != 1) && c->ny < G) return false;
    if (c->time_scheme != DFGKS_TIME_S2O4) return false;
    return (c->tau_reading == 0 || c->tau_reading == 1) && (c->dt_rule == 0 || c->dt_rule == 1)
        && (c->df_states == 0 || c->df_states == 1) && c->alpha_source == 0;
}

void make_plan(const dfgks_config* c, int px, int py, int b, dfgks_block_plan* p) {
    const int bx = b % px, by = b / px;
    p->i0 = split(c->nx, px, bx); p->i1 = split(c->nx, px, bx + 1);
    p->j0 = split(c->ny, py, by); p->j1 = split(c->ny, py, by + 1);
    const int bc[4] = {c->bc_xlo, c->bc_xhi, c->bc_ylo, c->bc_yhi};
    // x-low, x-high, y-low, y-high: an inner side, or a periodic side of a split direction, is
    // shared with the neighbouring block; otherwise the side keeps the mesh's boundary condition
    const bool inner[4] = {bx > 0, bx < px - 1, by > 0, by < py - 1};
    const int wrap[4] = {by * px + px - 1, by * px, (py - 1) * px + bx, bx};
    const int next[4] = {b - 1, b + 1, b - px, b + px};
    const bool split_dir[4] = {px > 1, px > 1, py > 1, py > 1};
    for (int s = 0; s < 4; ++s) {
        if (inner[s]) { p->bc[s] = BC_EXTERNAL; p->neighbour[s] = next[s]; }
        else if (bc[s] == DFGKS_BC_PERIODIC && split_dir[s]) { p->bc[s] = BC_EXTERNAL; p->neighbour[s] = wrap[s]; }
        else { p->bc[s] = bc[s]; p->neighbour[s] = -1; }
    }
}

}  // namespace

struct dfgks_decomp {
    dfgks_config cfg;
    int px, py;
    cudaStream_t stream;
    bool own_stream;
    SchemeConsts S;
    std::vector<Block> blk;
    DevState* st;            // shared by all blocks
    DevState* st_host;
    int* flag;
    int* flag_host;
    double* dts;             // device dt history of one step call
    int dts_cap;
    double* one;             // device scalar 1.0 (the alpha^0 pass)
    double* stage;           // dense [4][ny][nx] of the whole mesh: transfers
    int cur;
    std::vector<void*> allocs;
    HaloBlock* halo;         // device
    int* hold;               // device: the halt flag as the stage's ghost fill saw it
    int halo_tiles[2];       // 128-thread tiles of the largest block's ghost cells per pass
    // Helpers: the blocks' kernels between two ghost fills are independent and a block alone leaves part of the
    // chip idle, so block b runs on stream b mod their number.  With the fused ghost fill, 4 steps of 3 x 2 blocks
    // of 100 x 100 11.8 -> 5.6 ms.
    std::vector<cudaStream_t> streams;
    std::vector<cudaEvent_t> done;
    cudaEvent_t ready;
};

static dfgks_status dstat(cudaError_t e) {
    return e == cudaSuccess ? DFGKS_OK : (e == cudaErrorMemoryAllocation ? DFGKS_ENOMEM : DFGKS_ECUDA);
}
#define DCK(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return dstat(e_); } while (0)

template <class T>
static cudaError_t dalloc(dfgks_decomp* d, T** p, long long n) {
    cudaError_t e = cudaMalloc((void**)p, (size_t)n * sizeof(T));
    if (e == cudaSuccess) d->allocs.push_back((void*)*p);
    return e;
}

static void free_decomp(dfgks_decomp* d) {
    for (void* p : d->allocs) cudaFree(p);
    if (d->st_host) cudaFreeHost(d->st_host);
    if (d->flag_host) cudaFreeHost(d->flag_host);
    for (cudaEvent_t e : d->done) cudaEventDestroy(e);
    if (d->ready) cudaEventDestroy(d->ready);
    for (cudaStream_t s : d->streams) cudaStreamDestroy(s);
    if (d->own_stream && d->stream) cudaStreamDestroy(d->stream);
}

// The halo copy of side `side` of block b from its neighbour a: the window of b's ghosted field
// it fills ((di, dj), w x h cells) and where that window starts in a's field ((si, sj)).  Pass 0
// (x sides): the ghost columns of the interior rows from a's G boundary columns; pass 1 (y sides):
// the ghost rows, ghost columns included, from a's G boundary rows (with a's ghost columns, so the
// diagonal neighbour's cells reach the corners).
static void halo_window(const dfgks_block_plan& b, const dfgks_block_plan& a, int side, dfgks_halo_window* w) {
    const int bnx = b.i1 - b.i0, bny = b.j1 - b.j0, anx = a.i1 - a.i0, any = a.j1 - a.j0;
    if (side < 2) {
        w->w = G; w->h = bny; w->dj = 0; w->sj = 0;
        if (side == 0) { w->di = -G; w->si = anx - G; } else { w->di = bnx; w->si = 0; }
    } else {
        w->w = bnx + 2 * G; w->h = G; w->di = -G; w->si = -G;
        if (side == 2) { w->dj = -G; w->sj = any - G; } else { w->dj = bny; w->sj = 0; }
    }
}

// ghost layers of every block: field 0 = W[in] (with alpha[in] when with_alpha), 1 = Ws
static cudaError_t halo(dfgks_decomp* d, int field, int in, bool with_alpha) {
    for (int pass = 0; pass < 2; ++pass)
        k_halo<<<dim3((unsigned)d->blk.size(), d->halo_tiles[pass]), 128, 0, d->stream>>>(
            d->halo, pass, field == 0 ? in : 2, with_alpha ? in : -1, &d->st->halt, d->hold);
    return cudaGetLastError();
}

// the blocks' streams after the handle's stream, and the handle's stream after theirs
static cudaError_t fork(dfgks_decomp* d) {
    cudaError_t e = d->streams.empty() ? cudaSuccess : cudaEventRecord(d->ready, d->stream);
    for (size_t q = 0; q < d->streams.size() && e == cudaSuccess; ++q) e = cudaStreamWaitEvent(d->streams[q], d->ready, 0);
    return e;
}
static cudaError_t join(dfgks_decomp* d) {
    cudaError_t e = cudaSuccess;
    for (size_t q = 0; q < d->streams.size() && e == cudaSuccess; ++q) {
        e = cudaEventRecord(d->done[q], d->streams[q]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(d->stream, d->done[q], 0);
    }
    return e;
}
static cudaStream_t stream_of(const dfgks_decomp* d, size_t b) { return d->streams.empty() ? d->stream : d->streams[b % d->streams.size()]; }

// blocks (all of about one size) whose kernels run side by side
static int blocks_beside(const dfgks_decomp* d) { return d->streams.empty() ? 1 : (int)d->streams.size(); }

static cudaError_t create_halo(dfgks_decomp* d) {
    std::vector<HaloBlock> H(d->blk.size());
    int rows = 0, cols = 0;
    for (size_t b = 0; b < H.size(); ++b) {
        const Block& k = d->blk[b];
        HaloBlock& h = H[b];
        h.m = k.m;
        h.W[0] = k.W[0]; h.W[1] = k.W[1]; h.W[2] = k.Ws; h.A[0] = k.A[0]; h.A[1] = k.A[1];
        for (int s = 0; s < 4; ++s) {
            dfgks_halo_window w = {};
            h.neighbour[s] = k.plan.neighbour[s];
            if (h.neighbour[s] >= 0) halo_window(k.plan, d->blk[h.neighbour[s]].plan, s, &w);
            h.di[s] = w.di; h.dj[s] = w.dj; h.si[s] = w.si; h.sj[s] = w.sj;
        }
        if (k.m.ny > rows) rows = k.m.ny;
        if (k.m.nx + 2 * G > cols) cols = k.m.nx + 2 * G;
    }
    d->halo_tiles[0] = (2 * G * rows + 127) / 128;
    d->halo_tiles[1] = (2 * G * cols + 127) / 128;
    cudaError_t e = dalloc(d, &d->halo, (long long)H.size());
    // on the handle's stream, which k_halo runs on: a plain cudaMemcpy goes to the legacy stream, may return before the
    // data has reached the device, and a non-blocking stream does not wait for it
    if (e == cudaSuccess) e = cudaMemcpyAsync(d->halo, H.data(), H.size() * sizeof(HaloBlock), cudaMemcpyHostToDevice, d->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(d->stream);          // H ends here
    const size_t n = H.size() < 2 ? 0 : (H.size() < 8 ? H.size() : 8);
    if (e == cudaSuccess && n) e = cudaEventCreateWithFlags(&d->ready, cudaEventDisableTiming);
    for (size_t q = 0; q < n && e == cudaSuccess; ++q) {
        cudaStream_t st;
        cudaEvent_t ev;
        if ((e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) == cudaSuccess) d->streams.push_back(st);
        if (e == cudaSuccess && (e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) == cudaSuccess) d->done.push_back(ev);
    }
    return e;
}

static dfgks_status reset_state(dfgks_decomp* d, double t, long long step) {
    DevState z;
    memset(&z, 0, sizeof(z));
    z.t = t;
    z.step = step;
    z.dtmin_bits = 0x7FEFFFFFFFFFFFFFULL;
    z.fail_step = -1;
    z.fail_key = ~0ULL;
    *d->st_host = z;
    DCK(cudaMemcpyAsync(d->st, d->st_host, sizeof(DevState), cudaMemcpyHostToDevice, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    return DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_plan(const dfgks_config* cfg, int px, int py, int block,
                                                    dfgks_block_plan* out) {
    if (!out || !decomp_config_ok(cfg, px, py) || block < 0 || block >= px * py) return DFGKS_EINVAL;
    make_plan(cfg, px, py, block, out);
    return DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_halo(const dfgks_config* cfg, int px, int py, int block, int side,
                                                    dfgks_halo_window* out) {
    if (!out || !decomp_config_ok(cfg, px, py) || block < 0 || block >= px * py || side < 0 || side > 3)
        return DFGKS_EINVAL;
    dfgks_block_plan b, a;
    make_plan(cfg, px, py, block, &b);
    out->neighbour = b.neighbour[side];
    if (out->neighbour < 0) { out->di = out->dj = out->si = out->sj = out->w = out->h = 0; return DFGKS_OK; }
    make_plan(cfg, px, py, out->neighbour, &a);
    halo_window(b, a, side, out);
    return DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_create(const dfgks_config* cfg, int px, int py, void* stream,
                                                      dfgks_decomp** out) {
    if (!out) return DFGKS_EINVAL;
    *out = nullptr;
    if (!decomp_config_ok(cfg, px, py)) return DFGKS_EINVAL;
    dfgks_decomp* d = new (std::nothrow) dfgks_decomp();
    if (!d) return DFGKS_ENOMEM;
    d->cfg = *cfg;
    d->px = px; d->py = py;
    d->st_host = nullptr; d->flag_host = nullptr;
    d->cur = 0;
    if (stream) { d->stream = (cudaStream_t)stream; d->own_stream = false; }
    else if (cudaStreamCreateWithFlags(&d->stream, cudaStreamNonBlocking) != cudaSuccess) { delete d; return DFGKS_ECUDA; }
    else d->own_stream = true;
    SchemeConsts& S = d->S;
    memset(&S, 0, sizeof(S));
    S.gamma = cfg->gamma; S.gm1 = cfg->gamma - 1.0; S.K = (4.0 - 2.0 * cfg->gamma) / (cfg->gamma - 1.0);
    S.inv_K2 = 1.0 / (S.K + 2.0);
    S.r2g = sqrt(2.0 / S.gamma);
    S.d[3] = cfg->dH; S.d[0] = (1.0 - cfg->dH) * (1.0 - cfg->dL) / 2.0; S.d[1] = (1.0 - cfg->dH) * cfg->dL; S.d[2] = S.d[0];
    S.inv_d3 = 1.0 / cfg->dH;
    S.eps = cfg->eps; S.alpha_thres = cfg->alpha_thres; S.C1 = cfg->C1; S.C2 = cfg->C2;
    S.time_limiter = cfg->time_limiter; S.tau_reading = cfg->tau_reading; S.gp_fallback = cfg->gp_fallback;
    S.df_states = cfg->df_states;
    const double dx = (cfg->x1 - cfg->x0) / cfg->nx, dy = (cfg->y1 - cfg->y0) / cfg->ny;
    cudaError_t e = cudaSuccess;
    long long cells = 0;
    d->blk.resize((size_t)px * py);
    for (int b = 0; b < px * py && e == cudaSuccess; ++b) {
        Block& k = d->blk[b];
        memset(&k, 0, sizeof(k));
        make_plan(cfg, px, py, b, &k.plan);
        Mesh& m = k.m;
        m.nx = k.plan.i1 - k.plan.i0; m.ny = k.plan.j1 - k.plan.j0;
        m.P = (int)round4(m.nx + 2 * G);
        m.NYg = m.ny + 2 * G;
        m.plane = (long long)m.P * m.NYg;
        m.dx = dx; m.dy = dy;
        m.rdx = 1.0 / dx; m.rdy = 1.0 / dy;
        for (int s = 0; s < 4; ++s) m.bc[s] = k.plan.bc[s];
        m.dt_rule = cfg->dt_rule;
        // a failing cell's key: the cells of the blocks before, then row by row in its block (failing_cell), so the
        // smallest key is in the first failing block.  (2^31 cells would take terabytes.)
        m.gi0 = (int)cells; m.gj0 = 0; m.gnx = m.nx;
        cells += (long long)m.nx * m.ny;
        const long long nfx = (long long)(m.nx + 1) * m.ny, nfy = (long long)(m.ny + 1) * m.nx;
        const long long nlx = (long long)(m.nx + 1) * (m.ny + 4), nly = (long long)(m.ny + 1) * (m.nx + 4);
        k.B.line_stride = round4(nlx > nly ? nlx : nly);
        k.B.gp_stride = round4(2 * (nfx > nfy ? nfx : nfy));
        k.B.flux_stride[0] = round4(2 * nfx);
        k.B.flux_stride[1] = round4(2 * nfy);
        if (e == cudaSuccess) e = dalloc(d, &k.W[0], 4 * m.plane);
        if (e == cudaSuccess) e = dalloc(d, &k.W[1], 4 * m.plane);
        if (e == cudaSuccess) e = dalloc(d, &k.A[0], m.plane);
        if (e == cudaSuccess) e = dalloc(d, &k.A[1], m.plane);
        if (e == cudaSuccess) e = dalloc(d, &k.Ws, 4 * m.plane);
        if (e == cudaSuccess) e = dalloc(d, &k.acc, 4LL * m.nx * m.ny);
        if (e == cudaSuccess) e = dalloc(d, &k.B.lines, (long long)LR_COUNT * k.B.line_stride);
        if (e == cudaSuccess) e = dalloc(d, &k.B.gp, (long long)GP_COUNT * k.B.gp_stride);
        if (e == cudaSuccess) e = dalloc(d, &k.B.flux[0], (long long)FR_COUNT * k.B.flux_stride[0]);
        if (e == cudaSuccess) e = dalloc(d, &k.B.flux[1], (long long)FR_COUNT * k.B.flux_stride[1]);
        k.By = k.B;
        if (e == cudaSuccess) e = dalloc(d, &k.By.lines, (long long)LR_COUNT * k.B.line_stride);
        if (e == cudaSuccess) e = dalloc(d, &k.By.gp, (long long)GP_COUNT * k.B.gp_stride);
        if (e == cudaSuccess) {
            launch_fill_value(k.W[0], 4 * m.plane, 1.0, d->stream);
            launch_fill_value(k.W[1], 4 * m.plane, 1.0, d->stream);
            launch_fill_value(k.Ws, 4 * m.plane, 1.0, d->stream);
            launch_fill_value(k.A[0], m.plane, 1.0, d->stream);
            launch_fill_value(k.A[1], m.plane, 1.0, d->stream);
        }
    }
    if (e == cudaSuccess) e = dalloc(d, &d->st, 1);
    if (e == cudaSuccess) e = dalloc(d, &d->flag, 1);
    if (e == cudaSuccess) e = dalloc(d, &d->hold, 1);
    if (e == cudaSuccess) { d->dts_cap = 1024; e = dalloc(d, &d->dts, d->dts_cap); }
    if (e == cudaSuccess) e = dalloc(d, &d->one, 4);
    if (e == cudaSuccess) e = dalloc(d, &d->stage, 4LL * cfg->nx * cfg->ny);
    if (e == cudaSuccess) e = cudaMallocHost((void**)&d->st_host, sizeof(DevState));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&d->flag_host, sizeof(int));
    if (e == cudaSuccess) e = create_halo(d);
    if (e == cudaSuccess) launch_set_scalar(d->one, 1.0, d->stream);
    dfgks_status r = dstat(e);
    if (r == DFGKS_OK) r = reset_state(d, 0.0, 0);
    if (r != DFGKS_OK) { free_decomp(d); delete d; return r; }
    *out = d;
    return DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_destroy(dfgks_decomp* d) {
    if (!d) return DFGKS_OK;
    cudaStreamSynchronize(d->stream);
    free_decomp(d);
    delete d;
    return DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_set_ic(dfgks_decomp* d, const double* W, int on_device) {
    if (!d || !W) return DFGKS_EINVAL;
    const int nx = d->cfg.nx, ny = d->cfg.ny;
    const long long N = (long long)nx * ny;
    DCK(cudaMemcpyAsync(d->stage, W, (size_t)(4 * N) * sizeof(double),
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, d->stream));
    DCK(cudaMemsetAsync(d->flag, 0, sizeof(int), d->stream));
    d->cur = 0;
    for (Block& b : d->blk) {
        const long long nb = (long long)b.m.nx * b.m.ny;
        for (int k = 0; k < 4; ++k)
            DCK(cudaMemcpy2DAsync(b.acc + k * nb, (size_t)b.m.nx * sizeof(double),
                                  d->stage + k * N + (long long)b.plan.j0 * nx + b.plan.i0, (size_t)nx * sizeof(double),
                                  (size_t)b.m.nx * sizeof(double), (size_t)b.m.ny, cudaMemcpyDeviceToDevice, d->stream));
        launch_dense_to_ghosted(b.m, b.acc, 4, b.W[0], d->stream);
        launch_check_state(b.m, b.W[0], d->S.gm1, d->flag, d->stream);
    }
    DCK(cudaGetLastError());
    DCK(cudaMemcpyAsync(d->flag_host, d->flag, sizeof(int), cudaMemcpyDeviceToHost, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    if (*d->flag_host) return DFGKS_ENONPHYS;
    // alpha^0: the Gauss-point DF factors of a reconstruction of W^0 with alpha = 1
    dfgks_status r = reset_state(d, 0.0, 0);
    if (r != DFGKS_OK) return r;
    for (Block& b : d->blk) launch_fill_value(b.A[0], b.m.plane, 1.0, d->stream);
    DCK(halo(d, 0, 0, false));
    DCK(fork(d));
    for (size_t q = 0; q < d->blk.size(); ++q) {
        Block& b = d->blk[q];
        launch_sweep_xy(b.m, d->S, 1, SWEEP_ALPHA, b.W[0], b.A[0], d->one, b.B, b.By, nullptr, nullptr, stream_of(d, q),
                        nullptr, blocks_beside(d));
        UpdateArgs a;
        memset(&a, 0, sizeof(a));
        a.alpha_out = b.A[0];
        launch_update(UM_ALPHA, b.m, d->S, a, b.B, d->one, nullptr, nullptr, stream_of(d, q));
    }
    DCK(join(d));
    DCK(cudaGetLastError());
    DCK(cudaStreamSynchronize(d->stream));
    return DFGKS_OK;
}

// one S2O4 step (Eq. 24 with the time limiter) of all blocks from buffer `in` to `in ^ 1`; every
// kernel returns at once once the shared halt flag is set, so a queue of steps drains without
// work and the state stays at the last good step
static cudaError_t enqueue_decomp_step(dfgks_decomp* d, int s, int in, int flux, double t_end) {
    cudaStream_t st = d->stream;
    DevState* ds = d->st;
    const int* halt = &ds->halt;
    const double* dtp = &ds->dt;
    const int out = in ^ 1;
    cudaError_t e = fork(d);
    if (e != cudaSuccess) return e;
    for (size_t q = 0; q < d->blk.size(); ++q)                                    // minimum over all blocks
        launch_cfl_min(d->blk[q].m, d->blk[q].W[in], d->S.gamma, ds, stream_of(d, q));
    if ((e = join(d)) != cudaSuccess) return e;
    launch_begin_step(ds, d->cfg.cfl, 0.0, t_end, d->dts, s, st);
    for (int stage = 0; stage < 2; ++stage) {
        e = halo(d, stage, in, stage == 0);
        if (e == cudaSuccess) e = fork(d);
        if (e != cudaSuccess) return e;
        for (size_t q = 0; q < d->blk.size(); ++q) {
            Block& b = d->blk[q];
            launch_sweep_xy(b.m, d->S, flux, SWEEP_FULL, stage == 0 ? b.W[in] : b.Ws, b.A[in], dtp, b.B, b.By, ds, halt,
                            stream_of(d, q), nullptr, blocks_beside(d));
        }
        // An update that loses positivity halts all that starts later.  The updates of one stage run side by side, so
        // they go by the flag as the stage's ghost fill saw it (d->hold): each of them looks at all its cells, and the
        // cell reported is the first one of the first failing block, whichever update came first.  None starts before
        // every sweep has ended, as those go by the flag itself.
        if ((e = join(d)) != cudaSuccess || (e = fork(d)) != cudaSuccess) return e;
        for (size_t q = 0; q < d->blk.size(); ++q) {
            Block& b = d->blk[q];
            UpdateArgs a;
            memset(&a, 0, sizeof(a));
            a.acc = b.acc;
            if (stage == 0) { a.Win = b.W[in]; a.Wout = b.Ws; }
            else { a.Win = b.Ws; a.Wout = b.W[out]; a.alpha_out = b.A[out]; }
            launch_update(stage == 0 ? UM_S2O4_1 : UM_S2O4_2, b.m, d->S, a, b.B, dtp, ds, d->hold, stream_of(d, q));
        }
        if ((e = join(d)) != cudaSuccess) return e;
    }
    launch_end_step(ds, t_end, st);
    return cudaGetLastError();
}

// n steps with the CFL dt (the minimum over all blocks), the last clipped to t_end > 0; one
// synchronisation at the end.  ENONPOS on a positivity failure (dfgks_decomp_status gives the cell
// in the whole mesh), with the state left at the last good step.
extern "C" DFGKS_API dfgks_status dfgks_decomp_step(dfgks_decomp* d, int n, int flux, double t_end, int* steps_done) {
    if (steps_done) *steps_done = 0;
    if (!d || n < 0 || (flux != DFGKS_FLUX_GKS && flux != DFGKS_FLUX_LF)) return DFGKS_EINVAL;
    if (n == 0) return DFGKS_OK;
    if (n > d->dts_cap) {
        double* p = nullptr;
        DCK(cudaMalloc((void**)&p, (size_t)n * sizeof(double)));
        d->allocs.push_back(p);
        d->dts = p;
        d->dts_cap = n;
    }
    DCK(cudaMemsetAsync(&d->st->halt, 0, sizeof(int), d->stream));
    DCK(cudaMemsetAsync(&d->st->err, 0, sizeof(int), d->stream));
    DCK(cudaMemcpyAsync(d->st_host, d->st, sizeof(DevState), cudaMemcpyDeviceToHost, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    const long long step0 = d->st_host->step;
    const int cur0 = d->cur;
    for (int s = 0; s < n; ++s) DCK(enqueue_decomp_step(d, s, (cur0 + s) & 1, flux, t_end));
    DCK(cudaMemcpyAsync(d->st_host, d->st, sizeof(DevState), cudaMemcpyDeviceToHost, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    const long long done = d->st_host->step - step0;
    d->cur = (int)((cur0 + done) & 1);
    if (steps_done) *steps_done = (int)done;
    return d->st_host->err ? DFGKS_ENONPOS : DFGKS_OK;
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_get_state(dfgks_decomp* d, double* W, double* alpha, double* t, long* step,
                                                         int on_device) {
    if (!d) return DFGKS_EINVAL;
    const int nx = d->cfg.nx;
    const long long N = (long long)nx * d->cfg.ny;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    for (int q = 0; q < 2; ++q) {
        double* dst = q == 0 ? W : alpha;
        if (!dst) continue;
        const int nc = q == 0 ? 4 : 1;
        for (Block& b : d->blk) {
            const long long nb = (long long)b.m.nx * b.m.ny;
            launch_ghosted_to_dense(b.m, q == 0 ? b.W[d->cur] : b.A[d->cur], nc, b.acc, d->stream);
            for (int k = 0; k < nc; ++k)
                DCK(cudaMemcpy2DAsync(d->stage + k * N + (long long)b.plan.j0 * nx + b.plan.i0, (size_t)nx * sizeof(double),
                                      b.acc + k * nb, (size_t)b.m.nx * sizeof(double), (size_t)b.m.nx * sizeof(double),
                                      (size_t)b.m.ny, cudaMemcpyDeviceToDevice, d->stream));
        }
        DCK(cudaGetLastError());
        DCK(cudaMemcpyAsync(dst, d->stage, (size_t)(nc * N) * sizeof(double), kind, d->stream));
    }
    DCK(cudaMemcpyAsync(d->st_host, d->st, sizeof(DevState), cudaMemcpyDeviceToHost, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    if (t) *t = d->st_host->t;
    if (step) *step = (long)d->st_host->step;
    return DFGKS_OK;
}

// the whole mesh's indices of the cell that a key names (Mesh::gi0)
static void failing_cell(const dfgks_decomp* d, unsigned long long key, int* i, int* j) {
    *i = *j = -1;
    for (const Block& b : d->blk) {
        const unsigned long long n = (unsigned long long)b.m.nx * b.m.ny;
        if (key < n) {
            *i = b.plan.i0 + (int)(key % (unsigned long long)b.m.nx);
            *j = b.plan.j0 + (int)(key / (unsigned long long)b.m.nx);
            return;
        }
        key -= n;
    }
}

extern "C" DFGKS_API dfgks_status dfgks_decomp_status(dfgks_decomp* d, int* err, int* fail_i, int* fail_j,
                                                      dfgks_counters* counters) {
    if (!d) return DFGKS_EINVAL;
    DCK(cudaMemcpyAsync(d->st_host, d->st, sizeof(DevState), cudaMemcpyDeviceToHost, d->stream));
    DCK(cudaStreamSynchronize(d->stream));
    const DevState& h = *d->st_host;
    if (err) *err = h.err;
    int i = -1, j = -1;
    if (h.err != 0) failing_cell(d, h.fail_key, &i, &j);
    if (fail_i) *fail_i = i;
    if (fail_j) *fail_j = j;
    if (counters) {
        counters->fallbacks = h.fallbacks;
        counters->df_normal = h.df_normal;
        counters->df_tangential = h.df_tangential;
    }
    return DFGKS_OK;
}
