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

// A call takes resident launches from this many steps on, where there is a
// plan for them.  Loading and storing the state costs 13 us (64 x 64) to 40 us
// (500 x 500) a call, the step saves 20 us (FP32 64 x 64), 5 us (FP32 256 x
// 256) or 18 us (FP64 500 x 500), but only 2 us for FP32 512 x 512: calls of 4
// steps are faster throughout in FP64 and up to 100 000 nodes in FP32 (20 us
// against 98 for 64 x 64, 28 against 43 for 256 x 256), larger FP32 lattices
// break even at about 20.
inline int resident_min(int prec, long long nodes)
{
    return prec == P_F64 || nodes <= 100000 ? 4 : 24;
}
// Autotuning times them over this many steps at least, whatever number it is
// asked for (per step they are compared with the tile kernels): the loading
// and storing of a call then counts as in the calls of a run, 0.2 to 0.6 us a
// step, and the least number of steps above is always reached.
constexpr int RESIDENT_TIMED = 64;
// Whether a lattice by itself that has a plan takes them without having been
// autotuned: all but a periodic FP32 one.  That is not for accuracy.  Any other
// order of sums moves the results of a phase separation from a uniform state,
// which such a lattice is often set up for and which amplifies every rounding:
// velocities of 387 x 171 after 342 steps 1.0e-4 (of their norm) from the 64 x
// 16 tiles', where either is 1.0 to 1.2e-4 from 64 bits.  A Simulation keeps
// the results it had there until it is autotuned.  A batch takes the resident
// steps on any lattice: its results there were never a Simulation's (its 32 x
// 32 tiles are 9e-5 from the 64 x 16 ones too), and the drops, slabs and walls
// of sweeps move by 1e-6; lbm_batch_set_tile keeps the tile kernels.
inline bool resident_alone(const Lattice &L) { return L.walls || L.precision == P_F64; }
// A launch takes at most this many, so that no kernel holds the GPU for long.
constexpr int RESIDENT_MAX = 4096;

struct ResidentPlan {
    std::vector<ResidentTile> tiles;  // one per CTA
    int w = 0, h = 0, gx = 0;
    int min_steps = 0;                // resident_min of all nodes
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
// Threads of the CTAs of tiles with more than 256 nodes.
constexpr int resident_threads(bool f64) { return f64 ? 384 : 512; }

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
