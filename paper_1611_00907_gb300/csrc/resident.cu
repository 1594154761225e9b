// Resident steps: cutting lattices into one rectangle per SM, and launching
// (the kernel is in resident_impl.cuh, one translation unit per precision).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>

#include "resident.h"

namespace cplbm {

cudaError_t launch_resident_f64(const ResidentArgs &a, bool batch, int grid, int threads,
                                size_t smem, cudaStream_t s);
cudaError_t launch_resident_f32(const ResidentArgs &a, bool batch, int grid, int threads,
                                size_t smem, cudaStream_t s);
cudaError_t launch_resident_f32off(const ResidentArgs &a, bool batch, int grid, int threads,
                                   size_t smem, cudaStream_t s);

namespace {

// ---------------------------------------------------------------------------
// Host: cutting lattices into tiles.
// ---------------------------------------------------------------------------
size_t tile_smem(int prec, int w, int h)
{
    return rho_bytes(prec) * (size_t)Geo(w, h).elems();
}

// Threads of a CTA: 256 while every node and every two rim nodes have one.
int rim_nodes(bool walls, int w, int h)
{
    const int side = walls ? HX : RIM;
    return 2 * RIM * (w + 2 * side) + 2 * side * h;
}
int threads_for(const Lattice &L, int w, int h)
{
    return w * h > 256 || rim_nodes(L.walls != 0, w, h) > 256 * RIM_NODES
               ? resident_threads(L.precision == P_F64) : 256;
}

// Cost of a step of a w x h tile on one SM.  FP64: instructions per node of
// the FP64 units, of which each quarter of the SM has one, so that four warps
// of nodes (128) cost as much as one node.  FP32: instructions issued per
// node and per node received.
double tile_cost(int prec, int w, int h)
{
    const double n = (double)w * h, m = (double)(w + 2) * (h + 2),
                 r = (double)(w + 4) * (h + 4), x = (double)(w + 6) * (h + 6);
    auto rounds = [](double v) { return 128 * std::ceil(v / 128); };
    if (prec == P_F64) return 85 * rounds(n) + 28 * rounds(m) + 8 * rounds(r);
    return 220 * n + 90 * m + 45 * r + 120 * (x - n);
}

// Cut an nx x ny (fluid) lattice into at most `most` tiles, the cheapest
// first: tile widths are multiples of four (the words of a rim row then fill
// whole 32-byte sectors), heights at least two; beside a wall no tile row is
// a single row, for the tile next to it would then need the solid row's
// density.  false when no cut fits shared memory.
bool cut(const Lattice &L, int most, int *w, int *h)
{
    const int prec = L.precision, nx = L.nx, ny = L.nyf;
    double best = -1;
    for (int ww = 4; ww < nx + 4; ww += 4) {
        const int cx = (nx + ww - 1) / ww;
        if (cx > most) continue;
        const int cy = std::min(most / cx, std::max(1, ny / 2));
        int hh = (ny + cy - 1) / cy;
        while (L.walls && ny % hh == 1) ++hh;
        const int tw = std::min(ww, nx);
        if (tile_smem(prec, tw, hh) > RESIDENT_SMEM ||
            rim_nodes(L.walls != 0, tw, hh) > resident_threads(prec == P_F64) * RIM_NODES)
            continue;
        const double c = tile_cost(prec, tw, hh);
        if (best < 0 || c < best) {
            best = c;
            *w = tw;
            *h = hh;
        }
    }
    return best >= 0;
}

int sm_count(int device)
{
    int n = 0, coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess ||
        !coop ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_prec(int prec, const ResidentArgs &a, bool batch, int grid, int threads,
                        size_t smem, cudaStream_t s)
{
    switch (prec) {
    case P_F64: return launch_resident_f64(a, batch, grid, threads, smem, s);
    case P_F32: return launch_resident_f32(a, batch, grid, threads, smem, s);
    case P_F32_OFF: return launch_resident_f32off(a, batch, grid, threads, smem, s);
    }
    return cudaErrorInvalidValue;
}

// Resident launches of one device follow one another whatever streams they
// are on: two of them, each holding a part of the SMs, would wait for the
// rest.  One event per device and CUDA context: a device reset ends both.
constexpr int MAX_DEVICES = 64;
struct Turn {
    std::mutex m;
    cudaEvent_t done = nullptr;
    unsigned long long ctx_id = 0;
};
Turn g_turn[MAX_DEVICES];

}  // namespace

size_t xchg_bytes(const Lattice &L)
{
    return 2 * 9 * (size_t)L.plane * 2 * rho_bytes(L.precision);
}

namespace {
bool make_plan(const Lattice *lats, int count, int device, ResidentPlan *p)
{
    if (count < 1 || device < 0 || device >= MAX_DEVICES) return false;
    const int prec = lats[0].precision;
    if (prec == P_F16_OFF) return false;
    // the largest state shared memory holds, before any search
    long long nodes = 0;
    for (int i = 0; i < count; ++i) nodes += (long long)lats[i].nx * lats[i].nyf;
    const int sms = sm_count(device);
    if (sms < 1 || count > sms ||
        nodes * 9 * (long long)rho_bytes(prec) > (long long)sms * (long long)RESIDENT_SMEM)
        return false;
    int wmax = 0, hmax = 0;
    std::vector<int> w(count), h(count);
    if (count == 1) {
        if (!cut(lats[0], sms, &w[0], &h[0])) return false;
    } else {
        // SMs shared out by nodes, the rest one by one to the lattice whose
        // tiles cost most
        std::vector<int> share(count);
        int used = 0;
        for (int i = 0; i < count; ++i) {
            const long long n = (long long)lats[i].nx * lats[i].nyf;
            share[i] = std::max(1, (int)(n * sms / nodes));
            used += share[i];
        }
        if (used > sms) return false;
        auto cost = [&](int i) {
            return cut(lats[i], share[i], &w[i], &h[i])
                       ? tile_cost(prec, w[i], h[i]) : 1e30;
        };
        std::vector<double> c(count);
        for (int i = 0; i < count; ++i) c[i] = cost(i);
        for (; used < sms; ++used) {
            const int i = (int)(std::max_element(c.begin(), c.end()) - c.begin());
            ++share[i];
            c[i] = cost(i);
        }
        if (*std::max_element(c.begin(), c.end()) >= 1e30) return false;
    }
    for (int i = 0; i < count; ++i) {
        wmax = std::max(wmax, w[i]);
        hmax = std::max(hmax, h[i]);
        p->smem = std::max(p->smem, tile_smem(prec, w[i], h[i]));
        for (int y = 0; y < lats[i].nyf; y += h[i])
            for (int x = 0; x < lats[i].nx; x += w[i])
                p->tiles.push_back({i, x, y, std::min(w[i], lats[i].nx - x),
                                    std::min(h[i], lats[i].nyf - y)});
        p->threads = std::max(p->threads, threads_for(lats[i], w[i], h[i]));
    }
    p->w = w[0];
    p->h = h[0];
    p->gx = (lats[0].nx + w[0] - 1) / w[0];
    p->min_steps = resident_min(prec, nodes);
    p->device = device;
    p->precision = prec;
    return (int)p->tiles.size() <= sms;
}
}  // namespace

// No exception leaves it (its callers are C entries): a host without memory
// for a plan steps on the tile kernels.
bool resident_plan(const Lattice *lats, int count, int device, ResidentPlan *p)
{
    *p = ResidentPlan{};
    try {
        if (make_plan(lats, count, device, p)) return true;
    } catch (const std::bad_alloc &) {
    }
    *p = ResidentPlan{};
    return false;
}

cudaError_t launch_resident(const ResidentPlan &p, const Lattice *single, const Lattice *d_lats,
                            const ResidentTile *d_tiles, int nsteps, int parity, unsigned tag,
                            cudaStream_t s)
{
    ResidentArgs a{};
    if (single) std::memcpy(&a.L, single, sizeof(Lattice));
    a.lats = d_lats;
    a.tiles = d_tiles;
    a.gx = p.gx;
    a.w = p.w;
    a.h = p.h;
    a.nsteps = nsteps;
    a.parity = parity;
    a.tag = tag;
    Turn &t = g_turn[p.device];
    std::lock_guard<std::mutex> lock(t.m);
    unsigned long long id = 0;
    current_context_id(&id);
    if (!t.done || t.ctx_id != id) {
        t.done = nullptr;
        cudaError_t e = cudaEventCreateWithFlags(&t.done, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            t.done = nullptr;
            return e;
        }
        t.ctx_id = id;
    } else {  // on the launch's own stream too: a stream's handle may be used again
        cudaError_t e = cudaStreamWaitEvent(s, t.done, 0);
        if (e != cudaSuccess) return e;
    }
    const int grid = (int)p.tiles.size();
    cudaError_t e = launch_prec(p.precision, a, single == nullptr, grid, p.threads, p.smem, s);
    // unrecorded, the event would let the next launch overlap this one
    if (e == cudaSuccess && cudaEventRecord(t.done, s) != cudaSuccess) e = cudaStreamSynchronize(s);
    return e;
}

}  // namespace cplbm
