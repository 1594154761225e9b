// Steps of small lattices with the state kept in shared memory
// (resident.cu): planning and launching.  Not public.
#pragma once

#include <cstring>
#include <vector>

#include "cplbm_internal.h"

namespace cplbm {

// The rectangle of one CTA: lattice `inst` of the launch, first node, size.
struct ResidentTile {
    int inst, x0, y0, w, h;
};

// Kernel parameter.  One lattice: L and its cut into tiles of w x h, gx to a
// row; several: descriptors and tiles in device memory.
struct ResidentArgs {
    Lattice L;
    const Lattice *lats;
    const ResidentTile *tiles;
    int gx, w, h;
    int nsteps, parity;   // steps of this call; parity of the first
    unsigned tag;         // tag of the first step's exchange words
};

// A call of at least RESIDENT_MIN steps takes resident launches where there
// is a plan for them; a launch takes at most RESIDENT_MAX, so that no kernel
// holds the GPU for long.
constexpr int RESIDENT_MIN = 4, RESIDENT_MAX = 4096;

struct ResidentPlan {
    std::vector<ResidentTile> tiles;  // one per CTA
    int w = 0, h = 0, gx = 0;
    int threads = 0;
    size_t smem = 0;
    int device = 0, precision = 0;
};

constexpr int RIM = 3;   // rows (columns) published along each tile edge
constexpr int HX = 4;    // columns of F beside the tile (one more beside a wall)

// Shared-memory geometry of a w x h tile (elements of the arithmetic type).
struct Geo {
    int w, h, fw, fp, rw, mw;
    __host__ __device__ Geo(int w_, int h_)
        : w(w_), h(h_), fw(w_ + 2 * HX), fp((w_ + 2 * HX) * (h_ + 2 * RIM)), rw(w_ + 6),
          mw(w_ + 2) {}
    // one row more than used in R and M: the second node of a row pair may
    // lie one row beyond them (computed, never stored)
    __host__ __device__ int elems() const { return 9 * fp + rw * (h + 5) + mw * (h + 3); }
};

constexpr size_t RESIDENT_SMEM = 220 * 1024;  // of 227 KB, beside the static part
constexpr int RIM_NODES = 2;   // rim nodes a thread receives at most

// Cut the lattices (of one precision) so that every tile has an SM of its
// own and fits its shared memory.  false when they are too large, too many,
// in FP16 storage, or the device has no cooperative launch.
bool resident_plan(const Lattice *lats, int count, int device, ResidentPlan *p);

// Bytes of a lattice's exchange words (Lattice::xchg), zeroed before use.
size_t xchg_bytes(const Lattice &L);

// Queue nsteps >= 2 steps from in-place parity `parity`.  single: the one
// lattice (d_lats, d_tiles unused), or null: descriptors and plan tiles in
// device memory.  Tags tag .. tag + nsteps - 1 must be new to the exchange
// words.
cudaError_t launch_resident(const ResidentPlan &p, const Lattice *single, const Lattice *d_lats,
                            const ResidentTile *d_tiles, int nsteps, int parity, unsigned tag,
                            cudaStream_t s);

}  // namespace cplbm
