// lpm_launch.h - host-side launch interface between the C-ABI layer and the kernels.
#pragma once

#include <nvtx3/nvToolsExt.h>

#include "lpm_device.cuh"

namespace lpm {

// A named NVTX range over a host scope (the enqueueing of a phase's device work: release,
// step, sort, advance, the adjoint's passes), for timeline tools; without a tool attached
// the push and pop return at once.
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// The device's error word and a page-locked host word: the kernels of a read-back copy the one to
// the other, so that one wait tells the error before anything goes to the caller's arrays, with
// no copy of its own (1e4 particles x 360 steps and their read-backs: 370 us with it, 358 without;
// the copies before the error is known 362).
struct ErrOut {
    const unsigned int *device;
    unsigned int *host;
};

// Counts of a sort: particles per key, and per tile of SCAN_TILE keys. Zero except between
// the pass that writes the keys and the sort that uses them up. Both padded to whole tiles.
constexpr int SCAN_TILE_BITS = 12;
constexpr int SCAN_TILE = 1 << SCAN_TILE_BITS;

struct SortCounts {
    unsigned int *keys, *tiles;
};

inline long long scan_tiles(long long n_keys) { return (n_keys + SCAN_TILE - 1) / SCAN_TILE; }

// The particles of an advance launch. A = the sorted live particles [0, live) of state_a
// (live count on the device; home slot of sorted slot i in pidx[i]; any scenario);
// B = tiles [b_first, b_first + n_b) of the tile table, each a run of one scenario's
// particles at their home slots in state_b.
struct Ranges {
    float4 *state_a;
    const unsigned int *a_live;   // nullptr: no particle has been sorted yet
    const unsigned int *pidx;
    float4 *state_b;
    const Tile *b_tiles;
    int b_first, n_b;
    int unit_shift;               // a B tile holds up to 32 << unit_shift particles
    unsigned int unit_min, unit_max;   // the launch runs if it has that many warps of particles
    float *w_a, *w_b;             // Langevin w' of A (sorted) and B (home) slots, or nullptr
    // when the next sort takes exactly this launch's particles as its inputs (A slots, then
    // the B tiles lane by lane): their sort keys and counts, written at the segment's end so
    // that the sort skips its key pass; else nullptr
    unsigned int *keys;
    SortCounts counts;
    int key_shift;
};

// Longest launch in steps: its step times sit in a table in shared memory.
constexpr int STEP_TAB = 128;

// AdvanceLaunch::occ of blocks whose warps work in pairs (256 threads, not the extended step),
// and the steps that one draws ahead for the other.
constexpr int OCC_PAIR = 3, PAIR_STEPS = 8;

// Options of an advance launch, by the instantiation that carries their code: none; the
// extended step (dosage, Eq. 3 K_z, a decay chain, the Langevin variant, with anything else);
// perturbation modes; a gridded K_h, the drift correction or levels without a lookup table;
// modes and any of these; the extended step on levels without a lookup table.
enum {
    ADV_PLAIN = 0,
    ADV_EXT = 1,
    ADV_MODES = 2,
    ADV_FIELDS = 3,
    ADV_MODES_FIELDS = 4,
    ADV_EXT_SEARCH = 5
};

constexpr bool adv_is_ext(int v) { return v == ADV_EXT || v == ADV_EXT_SEARCH; }

inline int adv_variant(const StepParams &P)
{
    if (P.dose_every > 0 || P.blpair || P.n_species > 1 || P.langevin)
        return P.lut_last < 0 ? ADV_EXT_SEARCH : ADV_EXT;
    const bool fields = P.khpair || P.drift || P.lut_last < 0;
    if (P.n_modes > 0) return fields ? ADV_MODES_FIELDS : ADV_MODES;
    return fields ? ADV_FIELDS : ADV_PLAIN;
}

struct AdvanceLaunch {
    cudaStream_t stream;
    const StepParams *params;
    Ranges ranges;
    unsigned int *queue;      // work-queue counter (zeroed before the launch)
    int k0, k1, do_bin;
    int block, occ;
    bool mixed;               // lanes of one tile may belong to different scenarios
    unsigned int grid;
    int variant() const { return adv_variant(*params); }
};

// Inputs of a sort: the live sorted particles of state_a (when has_a) followed by the B
// tiles [b_first, b_first + n_b) of the table at their home slots in state_b, T lanes each.
struct SortSource {
    const float4 *state_a;
    const unsigned int *pidx_a;
    bool has_a;
    long long a_bound;            // upper bound of the live count
    const float4 *state_b;
    const Tile *tiles;
    int b_first, n_b, t_shift;    // T = 1 << t_shift
    const float *w_a, *w_b;       // Langevin w' (moved with the particles), or nullptr
    bool keys_ready;              // keys and counts already written (fused key pass)
    int key_shift;                // cell keys are cell_key >> key_shift
    int key_scen;                 // 0: cell keys; n > 0: keys (scenario, cell tile) over n
                                  // scenarios, scenario-major (sort_dead_key)
};

struct SortBuffers {
    float4 *state_out;
    unsigned int *pidx_out;
    unsigned int *slot_of;        // per home slot: sorted slot, GRAVE | index, or SLOT_HOME;
                                  // nullptr: not kept (launch_slot_map rebuilds it)
    unsigned int *grave_home;     // home slot of each dead-particle entry, or nullptr
    unsigned int *keys, *offsets, *meta;   // offsets: first place of each key
    SortCounts counts;
    float4 *grave;
    unsigned int *grave_count;
    float *w_out;                 // Langevin w' of the sorted particles, or nullptr
    long long cap;                // entries of state_out, pidx_out, slot_of and grave
    unsigned int *err;            // device error word (bounds of the checked build)
};

// Sort keys: cells grouped in tiles of 2^SORT_TILE_BITS x 2^SORT_TILE_BITS columns by
// 2^SORT_TILE_ZBITS levels, tile by tile along x, then y, then z; keys run over
// [0, sort_key_range).
constexpr int SORT_TILE_BITS = 2;
constexpr int SORT_TILE_ZBITS = 2;

__host__ __device__ inline long long sort_key_range(int nx, int ny, int nz)
{
    const long long t = 1LL << SORT_TILE_BITS, tz = 1LL << SORT_TILE_ZBITS;
    return ((nz + tz - 1) / tz) * tz * ((ny + t - 1) / t) * ((nx + t - 1) / t) * t * t;
}

constexpr unsigned int KEY_NONE_U = 0xffffffffu;     // sort input that is no particle

// Key of the particles that left the working set (the last key of a sort): after the cell
// keys, or after key_scen scenarios' tile keys (scenario s, tile t: s * tiles + t, one
// key per tile of 2^(2 SORT_TILE_BITS + SORT_TILE_ZBITS) cells).
constexpr int SORT_CELL_BITS = 2 * SORT_TILE_BITS + SORT_TILE_ZBITS;   // cells of a tile, log2

__host__ __device__ inline long long sort_dead_key(int nx, int ny, int nz, int key_shift,
                                                   int key_scen)
{
    const long long r = sort_key_range(nx, ny, nz);
    return key_scen > 0 ? (long long)key_scen * (r >> SORT_CELL_BITS) : r >> key_shift;
}

// Cell keys of a sort of at most n particles: whole cells, or cell tiles where there are few
// particles a tile anyway (their order within it is of no use, and 64 times fewer keys are
// counted and scanned).
inline int sort_key_shift(long long n) { return n <= (1 << 17) ? SORT_CELL_BITS : 0; }

// Counts a key (KEY_NONE_U: none), one atomic per key and per tile of keys present in the
// warp. Every lane of the warp must call it.
__device__ __forceinline__ void sort_count(const SortCounts &C, unsigned int key)
{
    const int lane = threadIdx.x & 31;
    const unsigned int peers = __match_any_sync(0xffffffffu, key);
    if (key != KEY_NONE_U && lane == __ffs(peers) - 1)
        atomicAdd(C.keys + key, (unsigned int)__popc(peers));
    const unsigned int tile = key != KEY_NONE_U ? key >> SCAN_TILE_BITS : KEY_NONE_U;
    const unsigned int near = __match_any_sync(0xffffffffu, tile);
    if (tile != KEY_NONE_U && lane == __ffs(near) - 1)
        atomicAdd(C.tiles + tile, (unsigned int)__popc(near));
}

// Key of cell (ix, jy, kz): its tile, then its place in the tile.
__device__ __forceinline__ unsigned int cell_key(const StepParams &P, int ix, int jy, int kz)
{
    constexpr int TB = SORT_TILE_BITS, TZ = SORT_TILE_ZBITS;
    constexpr int T = 1 << TB, TZN = 1 << TZ;
    const unsigned int ntx = (unsigned int)((P.nx + T - 1) >> TB);
    const unsigned int nty = (unsigned int)((P.ny + T - 1) >> TB);
    const unsigned int tile = ((unsigned int)(kz >> TZ) * nty + (unsigned int)(jy >> TB)) * ntx +
                              (unsigned int)(ix >> TB);
    return (tile << (2 * TB + TZ)) | ((unsigned int)(kz & (TZN - 1)) << (2 * TB)) |
           ((unsigned int)(jy & (T - 1)) << TB) | (unsigned int)(ix & (T - 1));
}

constexpr unsigned int SLOT_HOME = 0xffffffffu;   // slot_of: the particle is at its home slot
constexpr unsigned int SLOT_GRAVE = 0x80000000u;  // slot_of flag: index into the dead array

// slot_of for every home slot [0, n_slots): SLOT_HOME, then the sorted slot of each of the
// meta[0] live particles (pidx: sorted slot -> home slot) and GRAVE | index of each of the
// *grave_n dead ones (grave_home: index -> home slot).
cudaError_t launch_slot_map(cudaStream_t s, const unsigned int *pidx, const unsigned int *meta,
                            const unsigned int *grave_home, const unsigned int *grave_n,
                            unsigned int *slot_of, long long n_slots, unsigned int *err);
cudaError_t launch_release(cudaStream_t s, float4 *state, long long first_slot, long long count,
                           long long part_first, long long n_total, int rel_first, int rel_len,
                           float sx, float sy, float sz);
cudaError_t launch_release_all(cudaStream_t s, const StepParams &P, float4 *state, long long n_slots);
// Bytes of dynamic shared memory of an advance launch: its level tables.
inline size_t adv_dyn_smem(int nz, int n_lut)
{
    return (size_t)nz * sizeof(float4) + (((size_t)(n_lut > 0 ? n_lut : 0) + 15) & ~(size_t)15);
}

cudaError_t launch_advance(const AdvanceLaunch &L);
int advance_occupancy(int block, int occ, bool mixed, int variant, size_t smem);
cudaError_t launch_advance_b128(const AdvanceLaunch &L);
cudaError_t launch_advance_b256(const AdvanceLaunch &L);
cudaError_t launch_advance_pair(const AdvanceLaunch &L);
cudaError_t launch_advance_b512(const AdvanceLaunch &L);
int occupancy_b128(int occ, bool mixed, int variant, size_t smem);
int occupancy_b256(int occ, bool mixed, int variant, size_t smem);
int occupancy_pair(bool mixed, int variant, size_t smem);
int occupancy_b512(int occ, bool mixed, int variant, size_t smem);
cudaError_t launch_pack(cudaStream_t s, const float4 *a, const float4 *b, const float *ka,
                        const float *kb, float4 *pair, float2 *khpair, int nx, int ny, int nz);
cudaError_t launch_pack_columns(cudaStream_t s, const float4 *a, const float4 *b, float4 *pair,
                                int nx, int ny);
cudaError_t launch_sort(cudaStream_t s, const StepParams &P, const SortSource &in,
                        const SortBuffers &out);
cudaError_t launch_gather(cudaStream_t s, const float4 *home, const float4 *sorted,
                          const unsigned int *slot_of, const float4 *grave, long long first,
                          long long count, float4 *out);
cudaError_t launch_gather_xyz(cudaStream_t s, const float4 *home, const float4 *sorted,
                              const unsigned int *slot_of, const float4 *grave, long long first,
                              long long count, float *xyz, unsigned int *tag, ErrOut err);
cudaError_t launch_gather_w(cudaStream_t s, const float *home, const float *sorted,
                            const unsigned int *slot_of, long long first, long long count,
                            float *out);
cudaError_t launch_unsort(cudaStream_t s, float4 *home, const float4 *sorted,
                          unsigned int *slot_of, const float4 *grave, long long n, float *w_home,
                          const float *w_sorted);
cudaError_t launch_draws(cudaStream_t s, unsigned long long seed, const unsigned long long *pid,
                         const unsigned int *step, unsigned int stream, long long n, uint4 *words,
                         float *nrm);
cudaError_t launch_budget(cudaStream_t s, const StepParams &P, const float4 *home, long long n_home,
                          const unsigned int *slot_of, const float4 *sorted,
                          const unsigned int *pidx, const unsigned int *live, long long a_bound,
                          int k_now);

cudaError_t launch_fixed_to_double(cudaStream_t s, const unsigned long long *in, double *out,
                                   long long n, double f, double d, ErrOut err);
void set_global_error(const char *msg);

struct AdjParams;
struct AdjSeg;
cudaError_t launch_adj_forward(cudaStream_t s, const StepParams &P, const AdjParams &A, int n_tiles);
cudaError_t launch_adj_backward(cudaStream_t s, const StepParams &P, const AdjParams &A, int n_tiles);
cudaError_t launch_adj_forward_seg(cudaStream_t s, const StepParams &P, const AdjParams &A,
                                   const AdjSeg &G, int n_groups, int mode, int n_sm);
cudaError_t launch_adj_backward_seg(cudaStream_t s, const StepParams &P, const AdjParams &A,
                                    const AdjSeg &G, int n_groups, int n_sm);

}  // namespace lpm
