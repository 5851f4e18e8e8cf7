/* C ABI of the batched 2D mode (gks_batch_*): many independent grids of
 * uneven sizes, kernels over tile work lists spanning every grid, per-grid time
 * steps on the device, one step captured into a CUDA graph and replayed.  Each
 * stage runs the three kernel classes of the single-grid step path
 * (reconstruction, face flux, update), one block per tile.  The wave-speed
 * kernel's tile and block size are picked by timing the candidates on the
 * actual grids before the graph is recorded, and cached per (dimension,
 * precision, size class of the batch, SM count), in the process and, if the
 * environment variable GKS_TUNE_CACHE names a file, in that file (one JSON
 * object per line), so a batch of the same size class skips the timing. */
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <algorithm>
#include <string>
#include <vector>

#include "batch.h"
#include "state_io.cuh"
#include "step_flux.cuh"

using gks::BatchLaunch;
using gks::GridDesc;
using gks::LaunchShape;
using gks::Tile;

struct gks_batch_ctx {
    int nb, precision;
    double gamma;
    int bc;
    gks_opts_t opts;
    cudaStream_t stream;      /* internal, capturable */
    cudaStream_t user_stream; /* ordering with the caller */
    cudaEvent_t ev_in, ev_out;
    std::vector<GridDesc> hd;
    GridDesc *dd;
    void *ws;
    size_t ws_bytes;
    double *dt;
    unsigned long long *smax;
    int *status; /* per-grid status words status[g] (OR of the ST_* bits) */
    float *updc; /* mixed precision: per-grid stage constants (UpdC, 10 floats each) */
    Tile *tiles[gks::BK_COUNT];
    int ntiles[gks::BK_COUNT];
    LaunchShape shape[gks::BK_COUNT];
    int tuned;
    /* mixed precision: per grid, gradients held only in the FP32 shadow
     * since the last run (G is filled from it when the state is read) */
    std::vector<char> g_stale;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    double graph_cfl;
    int nsm;
    char tuning[768];
    char err[256];
};

namespace {

thread_local char g_batch_err[256] = "";

int bfail(gks_batch_ctx *b, int code, const char *fmt, ...)
{
    char *buf = b ? b->err : g_batch_err;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, 256, fmt, ap);
    va_end(ap);
    return code;
}

int bcuda(gks_batch_ctx *b, cudaError_t e, const char *where)
{
    return bfail(b, GKS_ERR_CUDA, "%s: %s", where, cudaGetErrorString(e));
}

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

void make_kp(gks::KP &P, int nx, int ny, double h, double gamma, int bc, const gks_opts_t &o)
{
    std::memset(&P, 0, sizeof(P));
    P.n[0] = nx;
    P.n[1] = ny;
    P.n[2] = 1;
    P.ext[0] = nx + 2;
    P.ext[1] = ny + 2;
    P.ext[2] = 1;
    P.ncell = (long)nx * ny;
    P.next = (long)(nx + 2) * (ny + 2);
    P.nface[0] = (long)(nx + 1) * ny;
    P.nface[1] = (long)nx * (ny + 1);
    P.foff[0] = 0;
    P.foff[1] = P.nface[0];
    P.nftot = P.nface[0] + P.nface[1];
    gks::set_bcs(P, bc);
    P.limiter = o.limiter;
    P.h = h;
    P.ih = 1.0 / h;
    P.gamma = gamma;
    P.C = o.C;
    P.itanhC = 1.0 / std::tanh(o.C);
    P.eps = o.eps;
    P.C0 = o.C0;
    P.adm = o.adm_delta;
    P.d0 = o.ao_d0;
    P.ct = o.teno_ct;
    P.fp.gamma = gamma;
    P.fp.c1 = o.c1_tau;
    P.fp.c2 = o.c2_tau;
    gks::finalize_kp(P);
}

/* item count of kernel class k on grid g (flux: per direction) */
long items(const gks::KP &P, int k, int dir)
{
    switch (k) {
    case gks::BK_SPEED:
    case gks::BK_UPDATE: return P.ncell;
    case gks::BK_POLY: return P.next;
    default: return P.nface[dir];
    }
}

int build_tiles(gks_batch_ctx *b, int k, long tile)
{
    /* the previous list may still be read by work on the internal stream */
    cudaError_t se = cudaStreamSynchronize(b->stream);
    if (se != cudaSuccess) return bcuda(b, se, "tile list");
    std::vector<Tile> v;
    for (int g = 0; g < b->nb; ++g) {
        const gks::KP &P = b->hd[g].P;
        const int ndir = (k == gks::BK_FLUX) ? 2 : 1;
        for (int d = 0; d < ndir; ++d) {
            const long n = items(P, k, d);
            for (long s = 0; s < n; s += tile) v.push_back(Tile{2u * (unsigned)g + (unsigned)d, (unsigned)s});
        }
    }
    if (b->tiles[k]) cudaFree(b->tiles[k]);
    b->tiles[k] = nullptr;
    cudaError_t e = cudaMalloc(&b->tiles[k], sizeof(Tile) * v.size());
    if (e == cudaSuccess) e = cudaMemcpy(b->tiles[k], v.data(), sizeof(Tile) * v.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return bcuda(b, e, "tile list");
    b->ntiles[k] = (int)v.size();
    b->shape[k].tile = tile;
    return GKS_OK;
}

BatchLaunch launch_of(gks_batch_ctx *b, int k)
{
    return BatchLaunch{b->dd, b->tiles[k], b->ntiles[k], b->dt, b->updc, b->smax, b->status, &b->hd[0].P};
}

cudaError_t run_class(gks_batch_ctx *b, int k, int stage)
{
    const BatchLaunch L = launch_of(b, k);
    const LaunchShape &S = b->shape[k];
    const bool f = b->precision == 1;
    switch (k) {
    case gks::BK_SPEED: return f ? gks::batch_speed<float>(L, S, b->stream) : gks::batch_speed<double>(L, S, b->stream);
    case gks::BK_POLY: return f ? gks::batch_poly<float>(L, S, stage, b->stream) : gks::batch_poly<double>(L, S, stage, b->stream);
    case gks::BK_FLUX: return f ? gks::batch_flux<float>(L, S, stage, b->stream) : gks::batch_flux<double>(L, S, stage, b->stream);
    case gks::BK_UPDATE: return f ? gks::batch_update<float>(L, S, stage, b->stream) : gks::batch_update<double>(L, S, stage, b->stream);
    default: break;
    }
    /* BK_STAGE: a whole stage */
    for (int kk : {gks::BK_POLY, gks::BK_FLUX, gks::BK_UPDATE}) {
        const cudaError_t e = run_class(b, kk, stage);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

/* Launch shape of class k.  Stage kernels: one block per tile, one item per
 * thread (block threads a tile).  Wave speed: tiles of `tile` cells walked by
 * a persistent grid of the resident blocks. */
int set_shape(gks_batch_ctx *b, int k, int block, long tile)
{
    if (k == gks::BK_STAGE) {
        for (int kk : {gks::BK_POLY, gks::BK_FLUX, gks::BK_UPDATE}) {
            int r = set_shape(b, kk, 0, 0);
            if (r) return r;
        }
        b->shape[k] = b->shape[gks::BK_FLUX];
        return GKS_OK;
    }
    if (k != gks::BK_SPEED) tile = block = (k == gks::BK_FLUX) ? gks::kStepFluxBlock : 128;
    int r = build_tiles(b, k, tile);
    if (r) return r;
    const int occ = (k == gks::BK_SPEED) ? gks::batch_occupancy(b->precision, block) : 0;
    b->shape[k] = LaunchShape{block, tile, k == gks::BK_SPEED ? b->nsm * (occ > 0 ? occ : 1) : b->ntiles[k]};
    return GKS_OK;
}

/* one full step on the internal stream */
int enqueue_step(gks_batch_ctx *b, double cfl)
{
    cudaError_t e = cudaMemsetAsync(b->smax, 0, sizeof(unsigned long long) * b->nb, b->stream);
    if (e == cudaSuccess) e = run_class(b, gks::BK_SPEED, 1);
    if (e == cudaSuccess) e = gks::batch_dt(b->dd, b->nb, cfl, b->smax, b->dt, b->updc, b->stream);
    for (int stage = 1; stage <= 2 && e == cudaSuccess; ++stage) e = run_class(b, gks::BK_STAGE, stage);
    return e == cudaSuccess ? GKS_OK : bcuda(b, e, "batched step");
}

/* time one launch of class k (after one untimed launch) */
float time_class(gks_batch_ctx *b, int k)
{
    cudaEvent_t a, z;
    cudaEventCreate(&a);
    cudaEventCreate(&z);
    run_class(b, k, 1);
    cudaEventRecord(a, b->stream);
    run_class(b, k, 1);
    cudaEventRecord(z, b->stream);
    cudaEventSynchronize(z);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, a, z);
    cudaEventDestroy(a);
    cudaEventDestroy(z);
    return ms;
}

/* The kernel classes a batch reports: the wave speed, which is tuned, and the
 * three stage kernels, one by one in FP64 and as one entry in mixed precision. */
std::vector<int> classes_of(const gks_batch_ctx *b)
{
    if (b->precision == 1) return {gks::BK_SPEED, gks::BK_STAGE};
    return {gks::BK_SPEED, gks::BK_POLY, gks::BK_FLUX, gks::BK_UPDATE};
}

const char *class_name(int k)
{
    static const char *names[] = {"speed", "poly", "flux", "update", "stage"};
    return names[k];
}

/* Size class of a batch: powers of two of the grid count, of the total cell
 * count and of the largest side, with the dimension, precision, limiter
 * the device's SM count and the face flux's block size (a cache file written
 * for other kernels is not used). */
std::string size_class(const gks_batch_ctx *b)
{
    long cells = 0;
    int side = 0;
    for (int g = 0; g < b->nb; ++g) {
        cells += b->hd[g].P.ncell;
        side = std::max(side, std::max(b->hd[g].P.n[0], b->hd[g].P.n[1]));
    }
    auto lg = [](double x) { return (int)std::lround(std::log2(x > 1.0 ? x : 1.0)); };
    char k[160];
    snprintf(k, sizeof k, "2d/p%d/l%d/nb%d/cells%d/side%d/sm%d/t%d", b->precision, b->opts.limiter, lg(b->nb),
             lg((double)cells), lg(side), b->nsm, gks::kStepFluxBlock);
    return k;
}

struct TuneEntry {
    LaunchShape shape[gks::BK_COUNT];
};

std::mutex g_tune_mu;
std::map<std::string, TuneEntry> g_tune_cache;
bool g_tune_file_read = false;

/* the cache file named by GKS_TUNE_CACHE: one object per line,
 * {"key": "...", "shapes": [[block, tile, blocks], ... per kernel class]} */
void tune_file_read()
{
    if (g_tune_file_read) return;
    g_tune_file_read = true;
    const char *path = std::getenv("GKS_TUNE_CACHE");
    if (!path || !*path) return;
    FILE *f = std::fopen(path, "r");
    if (!f) return;
    char line[1024];
    while (std::fgets(line, sizeof line, f)) {
        const char *kp = std::strstr(line, "\"key\": \"");
        const char *sp = std::strstr(line, "\"shapes\": [");
        if (!kp || !sp) continue;
        kp += 8;
        const char *ke = std::strchr(kp, '"');
        if (!ke) continue;
        TuneEntry t;
        const char *q = sp + 11;
        bool ok = true;
        for (int k = 0; k < gks::BK_COUNT && ok; ++k) {
            long v[3];
            for (int j = 0; j < 3 && ok; ++j) {
                while (*q && (*q < '0' || *q > '9') && *q != '-') ++q;
                char *end = nullptr;
                v[j] = std::strtol(q, &end, 10);
                ok = end != q;
                q = end;
            }
            if (ok) t.shape[k] = LaunchShape{(int)v[0], v[1], (int)v[2]};
        }
        if (ok) g_tune_cache[std::string(kp, ke)] = t;
    }
    std::fclose(f);
}

void tune_file_append(const std::string &key, const TuneEntry &t)
{
    const char *path = std::getenv("GKS_TUNE_CACHE");
    if (!path || !*path) return;
    FILE *f = std::fopen(path, "a");
    if (!f) return;
    std::fprintf(f, "{\"key\": \"%s\", \"shapes\": [", key.c_str());
    for (int k = 0; k < gks::BK_COUNT; ++k)
        std::fprintf(f, "%s[%d, %ld, %d]", k ? ", " : "", t.shape[k].block, t.shape[k].tile, t.shape[k].blocks);
    std::fprintf(f, "]}\n");
    std::fclose(f);
}

/* Autotuner of the wave-speed kernel: tile size x block size candidates,
 * persistent grid = SMs x resident blocks; keep the fastest.  The stage
 * kernels' shapes are fixed (set_shape).  Runs only the wave speed (and its
 * time steps), so the state is unchanged.  A batch of a size class tuned
 * before (in this process or in the GKS_TUNE_CACHE file) takes the cached
 * shape without timing. */
int tune(gks_batch_ctx *b)
{
    const std::string key = size_class(b);
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        tune_file_read();
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            const LaunchShape &sp = it->second.shape[gks::BK_SPEED];
            int r = set_shape(b, gks::BK_SPEED, sp.block, sp.tile);
            if (r) return r;
            int pos = snprintf(b->tuning, sizeof(b->tuning), "{\"cached\": true, \"key\": \"%s\"", key.c_str());
            for (int k : classes_of(b))
                pos += snprintf(b->tuning + pos, sizeof(b->tuning) - pos, ", \"%s\": {\"block\": %d, \"tile\": %ld, \"blocks\": %d}",
                                class_name(k), b->shape[k].block, b->shape[k].tile, b->shape[k].blocks);
            snprintf(b->tuning + pos, sizeof(b->tuning) - pos, "}");
            b->tuned = 1;
            return GKS_OK;
        }
    }
    const long tiles[] = {512, 2048, 8192, 32768};
    int pos = 0;
    pos += snprintf(b->tuning + pos, sizeof(b->tuning) - pos, "{\"cached\": false, \"key\": \"%s\"", key.c_str());
    float best = 1e30f;
    LaunchShape bs{128, tiles[0], b->nsm};
    for (int block : {128, 256}) {
        for (long t : tiles) {
            int r = set_shape(b, gks::BK_SPEED, block, t);
            if (r) return r;
            cudaMemsetAsync(b->smax, 0, sizeof(unsigned long long) * b->nb, b->stream);
            const float ms = time_class(b, gks::BK_SPEED);
            if (ms < best) {
                best = ms;
                bs = b->shape[gks::BK_SPEED];
            }
        }
    }
    int r = set_shape(b, gks::BK_SPEED, bs.block, bs.tile);
    if (r) return r;
    for (int k : classes_of(b)) {
        const LaunchShape &sp = b->shape[k];
        pos += snprintf(b->tuning + pos, sizeof(b->tuning) - pos, ", \"%s\": {\"block\": %d, \"tile\": %ld, \"blocks\": %d",
                        class_name(k), sp.block, sp.tile, sp.blocks);
        if (k == gks::BK_SPEED) pos += snprintf(b->tuning + pos, sizeof(b->tuning) - pos, ", \"ms\": %.4f", best);
        pos += snprintf(b->tuning + pos, sizeof(b->tuning) - pos, "}");
    }
    snprintf(b->tuning + pos, sizeof(b->tuning) - pos, "}");
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "tuning");
    b->tuned = 1;
    TuneEntry t;
    for (int k = 0; k < gks::BK_COUNT; ++k) t.shape[k] = b->shape[k];
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        if (g_tune_cache.emplace(key, t).second) tune_file_append(key, t);
    }
    return GKS_OK;
}

} // namespace

extern "C" {

int gks_batch_create(int nbatch, const int *nx, const int *ny, const double *hs, double gamma, gks_bc_t bc,
                     const gks_opts_t *opts, gks_batch_t *out)
{
    if (!out) return bfail(nullptr, GKS_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (nbatch < 1 || !nx || !ny || !hs) return bfail(nullptr, GKS_ERR_ARG, "nbatch >= 1 and size arrays required");
    if (!(gamma > 1.0) || (bc != GKS_BC_PERIODIC && bc != GKS_BC_TRANSMISSIVE && bc != GKS_BC_REFLECTIVE &&
                            bc != GKS_BC_NOSLIP))
        return bfail(nullptr, GKS_ERR_ARG, "invalid gamma or boundary condition");
    gks_opts_t o;
    gks_default_opts(&o);
    if (opts) o = *opts;
    if (o.precision != 0 && o.precision != 1) return bfail(nullptr, GKS_ERR_ARG, "precision must be 0 or 1");
    if (o.limiter < 0 || o.limiter > 3) return bfail(nullptr, GKS_ERR_ARG, "limiter must be 0..3");
    if (o.limiter >= 2 && (!(o.ao_d0 > 0.0) || !(o.ao_d0 < 1.0) || !(o.teno_ct > 0.0) || !(o.teno_ct < 1.0)))
        return bfail(nullptr, GKS_ERR_ARG, "ao_d0 and teno_ct must lie in (0, 1)");
    if (o.workspace) return bfail(nullptr, GKS_ERR_UNSUPPORTED, "batched mode allocates its own workspace");
    if (o.mu != 0.0) return bfail(nullptr, GKS_ERR_UNSUPPORTED, "batched mode solves the Euler equations only (mu = 0)");
    for (int g = 0; g < nbatch; ++g) {
        if (nx[g] < 1 || ny[g] < 1 || nx[g] > (1 << 20) || ny[g] > (1 << 20) || !(hs[g] > 0.0))
            return bfail(nullptr, GKS_ERR_ARG, "grid %d: invalid size or cell size", g);
        /* the kernels decompose indices in 32-bit arithmetic */
        const long ext = (long)(nx[g] + 2) * (ny[g] + 2);
        const long gx = ((long)(nx[g] + 1) * ny[g] * 2 + 127) / 128 * 128;
        const long gy = ((long)nx[g] * (ny[g] + 1) * 2 + 127) / 128 * 128;
        if (ext >= (1L << 32) || gx >= (1L << 32) || gy >= (1L << 32))
            return bfail(nullptr, GKS_ERR_UNSUPPORTED, "grid %d too large (an index space reaches 2^32)", g);
    }

    gks_batch_ctx *b = new (std::nothrow) gks_batch_ctx();
    if (!b) return bfail(nullptr, GKS_ERR_OOM, "host allocation");
    b->nb = nbatch;
    b->precision = o.precision;
    b->gamma = gamma;
    b->bc = (int)bc;
    b->opts = o;
    b->user_stream = (cudaStream_t)o.stream;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&b->nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        int r = bcuda(nullptr, e, "stream/event creation");
        delete b;
        return r;
    }
    const size_t rs = o.precision ? sizeof(float) : sizeof(double);
    b->hd.resize(nbatch);
    b->g_stale.assign(nbatch, 0);
    size_t off = al(sizeof(double) * 2 * nbatch) + al(sizeof(unsigned long long) * nbatch) +
                 al(sizeof(float) * 10 * nbatch) + al(sizeof(int) * nbatch);
    std::vector<size_t> base(nbatch);
    for (int g = 0; g < nbatch; ++g) {
        make_kp(b->hd[g].P, nx[g], ny[g], hs[g], gamma, (int)bc, o);
        const gks::KP &P = b->hd[g].P;
        base[g] = off;
        off += al(sizeof(double) * 4 * P.ncell) * 2 + al(sizeof(double) * 8 * P.ncell) +
               al(rs * gks::group_elems(P.next, gks::kCellFields<2>)) + al(rs * gks::group_elems(P.nftot, gks::kFaceFields<2>));
        if (o.precision == 1) off += 2 * al(sizeof(float) * 16 * P.ncell); /* shadows: hi, lo, g */
        else off += al(sizeof(double) * 4 * P.ncell) + al(sizeof(double) * 8 * P.ncell); /* Ws, Gs */
    }
    b->ws_bytes = off;
    e = cudaMalloc(&b->ws, off);
    if (e != cudaSuccess) {
        int r = bfail(nullptr, GKS_ERR_OOM, "cudaMalloc of %zu bytes: %s", off, cudaGetErrorString(e));
        cudaStreamDestroy(b->stream);
        delete b;
        return r;
    }
    char *w = (char *)b->ws;
    b->dt = (double *)w;
    b->smax = (unsigned long long *)(w + al(sizeof(double) * 2 * nbatch));
    b->updc = (float *)((char *)b->smax + al(sizeof(unsigned long long) * nbatch));
    b->status = (int *)((char *)b->updc + al(sizeof(float) * 10 * nbatch));
    for (int g = 0; g < nbatch; ++g) {
        GridDesc &D = b->hd[g];
        const gks::KP &P = D.P;
        size_t o2 = base[g];
        D.W = (double *)(w + o2); o2 += al(sizeof(double) * 4 * P.ncell);
        D.Acc = (double *)(w + o2); o2 += al(sizeof(double) * 4 * P.ncell);
        D.G = (double *)(w + o2); o2 += al(sizeof(double) * 8 * P.ncell);
        D.B = w + o2; o2 += al(rs * gks::group_elems(P.next, gks::kCellFields<2>));
        D.ff = w + o2; o2 += al(rs * gks::group_elems(P.nftot, gks::kFaceFields<2>));
        D.Ws = D.Gs = nullptr;
        D.s0 = D.s1 = gks::Shadow{nullptr, nullptr, nullptr};
        if (o.precision == 1) {
            float *a = (float *)(w + o2), *c2 = (float *)(w + o2 + al(sizeof(float) * 16 * P.ncell));
            D.s0 = gks::Shadow{a, a + 4 * P.ncell, a + 8 * P.ncell};
            D.s1 = gks::Shadow{c2, c2 + 4 * P.ncell, c2 + 8 * P.ncell};
        } else {
            D.Ws = (double *)(w + o2); o2 += al(sizeof(double) * 4 * P.ncell);
            D.Gs = (double *)(w + o2);
        }
    }
    e = cudaMalloc(&b->dd, sizeof(GridDesc) * nbatch);
    if (e == cudaSuccess) e = cudaMemcpy(b->dd, b->hd.data(), sizeof(GridDesc) * nbatch, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(b->ws, 0, off);
    if (e != cudaSuccess) {
        int r = bcuda(nullptr, e, "batch setup");
        gks_batch_destroy(b);
        return r;
    }
    for (int k : classes_of(b)) {
        int r = set_shape(b, k, 128, 4096);
        if (r) {
            std::memcpy(g_batch_err, b->err, sizeof(g_batch_err));
            gks_batch_destroy(b);
            return r;
        }
    }
    *out = b;
    return GKS_OK;
}

int gks_batch_set_state(gks_batch_t b, int grid, const double *W, const double *G, int on_device)
{
    if (!b) return bfail(nullptr, GKS_ERR_ARG, "NULL handle");
    if (grid < 0 || grid >= b->nb || !W || !G) return bfail(b, GKS_ERR_ARG, "grid index or pointers invalid");
    const GridDesc &D = b->hd[grid];
    const size_t n = (size_t)4 * D.P.ncell;
    const cudaMemcpyKind k = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    /* the caller's buffers may still be written by work on its stream */
    cudaError_t e = cudaEventRecord(b->ev_in, b->user_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ev_in, 0);
    const bool direct = on_device && gks::in_device_memory(W, n * sizeof(double)) && gks::in_device_memory(G, 2 * n * sizeof(double));
    if (direct && e == cudaSuccess) e = gks::state_in<2>(W, G, D.W, D.G, D.s0, (long)n, b->status + grid, b->stream);
    if (!direct && e == cudaSuccess) e = cudaMemcpyAsync(D.W, W, n * sizeof(double), k, b->stream);
    if (!direct && e == cudaSuccess) e = cudaMemcpyAsync(D.G, G, 2 * n * sizeof(double), k, b->stream);
    if (!direct && e == cudaSuccess && b->precision == 1) e = gks::batch_shadow(D, b->stream);
    b->g_stale[grid] = 0;
    if (!direct && e == cudaSuccess) e = cudaMemsetAsync(b->status + grid, 0, sizeof(int), b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    return e == cudaSuccess ? GKS_OK : bcuda(b, e, "batch set_state");
}

int gks_batch_get_state(gks_batch_t b, int grid, double *W, double *G, int on_device)
{
    if (!b) return bfail(nullptr, GKS_ERR_ARG, "NULL handle");
    if (grid < 0 || grid >= b->nb) return bfail(b, GKS_ERR_ARG, "grid index invalid");
    const GridDesc &D = b->hd[grid];
    const size_t n = (size_t)4 * D.P.ncell;
    const cudaMemcpyKind k = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    /* the caller's stream may still use the destination buffers */
    cudaError_t e = cudaEventRecord(b->ev_in, b->user_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ev_in, 0);
    const bool direct = on_device && W && G && gks::in_device_memory(W, n * sizeof(double)) &&
                        gks::in_device_memory(G, 2 * n * sizeof(double));
    if (direct && e == cudaSuccess)
        e = gks::state_out<2>(D.W, D.G, b->precision && b->g_stale[grid] ? D.s0.g : nullptr, W, G, (long)n, b->stream);
    if (!direct && e == cudaSuccess && G && b->precision && b->g_stale[grid]) {
        e = gks::batch_widen_grad(D, b->stream);
        if (e == cudaSuccess) b->g_stale[grid] = 0;
    }
    if (!direct && e == cudaSuccess && W) e = cudaMemcpyAsync(W, D.W, n * sizeof(double), k, b->stream);
    if (!direct && e == cudaSuccess && G) e = cudaMemcpyAsync(G, D.G, 2 * n * sizeof(double), k, b->stream);
    int st = 0;
    if (e == cudaSuccess) e = gks::read_status(b->status + grid, &st, b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "batch get_state");
    if (st) return bfail(b, GKS_ERR_NONPHYSICAL, "grid %d: non-physical state (status bits 0x%x)", grid, st);
    return GKS_OK;
}

int gks_batch_run(gks_batch_t b, double cfl, int nsteps)
{
    if (!b) return bfail(nullptr, GKS_ERR_ARG, "NULL handle");
    if (!(cfl > 0.0) || !std::isfinite(cfl) || nsteps < 0) return bfail(b, GKS_ERR_ARG, "cfl > 0 and nsteps >= 0 required");
    if (b->precision == 1 && nsteps > 0) std::fill(b->g_stale.begin(), b->g_stale.end(), 1);
    cudaError_t e = cudaEventRecord(b->ev_in, b->user_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ev_in, 0);
    if (e != cudaSuccess) return bcuda(b, e, "stream ordering");
    if (!b->tuned) {
        int r = tune(b);
        if (r) return r;
    }
    if (!b->exec || b->graph_cfl != cfl) {
        if (b->exec) cudaGraphExecDestroy(b->exec);
        if (b->graph) cudaGraphDestroy(b->graph);
        b->exec = nullptr;
        b->graph = nullptr;
        e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return bcuda(b, e, "begin capture");
        int r = enqueue_step(b, cfl);
        cudaGraph_t g = nullptr;
        e = cudaStreamEndCapture(b->stream, &g);
        if (r) {
            if (g) cudaGraphDestroy(g);
            return r;
        }
        if (e != cudaSuccess) return bcuda(b, e, "end capture");
        b->graph = g;
        e = cudaGraphInstantiate(&b->exec, g, 0);
        if (e != cudaSuccess) return bcuda(b, e, "graph instantiate");
        b->graph_cfl = cfl;
    }
    for (int s = 0; s < nsteps; ++s) {
        e = cudaGraphLaunch(b->exec, b->stream);
        if (e != cudaSuccess) return bcuda(b, e, "graph launch");
    }
    e = cudaEventRecord(b->ev_out, b->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->user_stream, b->ev_out, 0);
    return e == cudaSuccess ? GKS_OK : bcuda(b, e, "stream ordering");
}

int gks_batch_status(gks_batch_t b)
{
    if (!b) return bfail(nullptr, GKS_ERR_ARG, "NULL handle");
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "stream synchronize");
    std::vector<int> st(b->nb);
    e = cudaMemcpy(st.data(), b->status, sizeof(int) * b->nb, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return bcuda(b, e, "status read");
    int r = 0;
    for (int v : st) r |= v;
    return r;
}

int gks_batch_grid_status(gks_batch_t b, int *status, int n)
{
    if (!b) return bfail(nullptr, GKS_ERR_ARG, "NULL handle");
    if (!status || n != b->nb) return bfail(b, GKS_ERR_ARG, "status must hold one word per grid (%d)", b->nb);
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "stream synchronize");
    e = cudaMemcpy(status, b->status, sizeof(int) * b->nb, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? GKS_OK : bcuda(b, e, "status read");
}

const char *gks_batch_tuning(gks_batch_t b) { return b ? b->tuning : ""; }

int gks_batch_destroy(gks_batch_t b)
{
    if (!b) return GKS_OK;
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (int k = 0; k < gks::BK_COUNT; ++k)
        if (b->tiles[k]) cudaFree(b->tiles[k]);
    if (b->dd) cudaFree(b->dd);
    if (b->ws) cudaFree(b->ws);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    if (b->ev_out) cudaEventDestroy(b->ev_out);
    if (b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return GKS_OK;
}

const char *gks_batch_last_error(gks_batch_t b) { return b ? b->err : g_batch_err; }

} // extern "C"
