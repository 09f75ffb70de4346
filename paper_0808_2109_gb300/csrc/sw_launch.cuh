// sw_launch.cuh -- how the host enqueues the kernels of sw_device.cuh: one
// launch group = the tile kernel of launch j, then the merge of sweep j.
// Shared by the single-lattice engine and the batch server.
#pragma once

#include "sw_device.cuh"

#include <cuda_runtime.h>

namespace swg {

// Defined once, in sw_engine.cu: every kernel template is instantiated in
// that translation unit only, so each kernel has a single module copy (and
// the shared-memory attribute set by prepare_th applies to the copy that
// runs).
__attribute__((visibility("hidden"))) cudaError_t prepare_th(int TH);
// feat: FEAT_* bits of the tile-kernel variant to launch (the union of what
// the launch's lattices need).  chained: the call's first kernel depends on the
// kernel before it in the stream as the others do on theirs (false: after
// memory operations, events or other kernels).
__attribute__((visibility("hidden"))) cudaError_t enqueue_tile(int TH, const SweepArgs &a, bool pcc, int feat,
                                                               cudaStream_t st, bool chained);
__attribute__((visibility("hidden"))) cudaError_t enqueue_merge(int TH, const SweepArgs &a, bool pcc, int feat,
                                                                cudaStream_t st, bool chained);
__attribute__((visibility("hidden"))) cudaError_t enqueue_launch_th(int TH, const SweepArgs &a, bool pcc, int feat,
                                                                    cudaStream_t st, bool chained);
// All sweeps of a one-tile lattice, L <= 128 (k_one), ONE_SWEEPS of them a launch
// (about 70 ms at L=128).
constexpr int32_t ONE_SWEEPS = 4096;
__attribute__((visibility("hidden"))) cudaError_t enqueue_one(const OneArgs &a, cudaStream_t st);
// Launch groups j = 0 .. m-1 of one lattice; last: the final one is a call's
// last and has no merge.
__attribute__((visibility("hidden"))) cudaError_t enqueue_groups(int TH, SweepArgs a, bool pcc, int feat, int m,
                                                                 bool last, cudaStream_t st);
__attribute__((visibility("hidden"))) cudaError_t enqueue_hot_start(uint8_t *spin, int64_t N, uint64_t seed,
                                                                    cudaStream_t st);
// One job, and n <= 65535 jobs of at most `most` items each (one launch).
__attribute__((visibility("hidden"))) cudaError_t enqueue_job_init(const JobInit &job, int64_t most, cudaStream_t st);
__attribute__((visibility("hidden"))) cudaError_t enqueue_jobs_init(const JobInit *jobs_dev, int n, int64_t most,
                                                                    cudaStream_t st);
__attribute__((visibility("hidden"))) cudaError_t enqueue_jobs_gather(const JobGather *jobs_dev, int n, int64_t most,
                                                                      cudaStream_t st);

// Whether a chain's kernels ask for the largest shared memory of an SM.  The split
// between it and the L1 cache changes only on an idle SM: left to itself, an SM with
// blocks of the merge kernels has room for no tile until they are gone, and the
// tiles started ahead crowd on the other SMs (every option at L=1920 65.4 us a sweep
// with the preference against 76.3).  The PCC kernels read through L1 (L=1001 46.9 us,
// with the preference 47.7), and so do the unions of the topological rule, which a grid
// of one wave does not crowd (L=800 46.4 either way); a grid that leaves half the GPU to
// its successors has nothing to gain (2D Potts L=64 16.5 either way).  For plain
// lattices the line was set on 64-row tiles (L=600 32 us against 43) and on Potts tiles
// of 8 warps (3D L=128 71 against 84), which those sizes no longer have: now L=600 to
// 2048 are within 1% either way, 2D Potts L=1024 takes 29.0 with the preference against
// 28.5 and 3D L=128 48.2 against 45.8, so that this part is due for another look.
inline bool chain_all_shared(int64_t n_tiles, bool pcc, bool wind)
{
    return !pcc && (wind ? n_tiles > FIRST_WAVE_SMS : 8 * n_tiles > FIRST_WAVE_SMS);
}

// Rows of a sub-tile of the 32-row tiles: 8 (16 warps a CTA) while there is at most
// one CTA an SM, 16 up to six, 32 beyond (8, 16 and 32 rows at T_c: L=300 22.2, 23.7
// and 27.3 us a sweep, L=700 24.0, 25.7 and 29.5, L=1400 36.9, 31.3 and 33.6, L=1920
// 45.4, 38.9 and 43.0, L=4096 153, 121 and 112; with cluster sizes L=300 27.6, 30.3 and
// 36.2).
inline int tile_rows(int n_tiles)
{
    return n_tiles <= FIRST_WAVE_SMS ? 8 : n_tiles <= 6 * FIRST_WAVE_SMS ? 16 : 32;
}

// Launches kernel k; chained: as a dependent of the kernel before it in the
// stream, which it may overlap (chain_next / chain_wait in sw_device.cuh).  The
// first kernel after anything else in the stream is not chained.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*k)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, bool chained,
                          bool all_shared, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    unsigned n = 0;
    if (all_shared) {
        at[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        at[n++].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    }
    if (chained) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

inline int slots_of(int TH) { return 2 * TW + 2 * TH; }

// A q-state Potts lattice on the d-dimensional lattice (sw_potts.cu): N =
// L^d sites cut into tiles (128 x 64 in 2D, 32 x 16 x 16 in 3D) of which the
// kernels keep per-tile scratch as the 2D Ising path does: a 2-byte code per
// site, crossing-bond bits and the face nodes' forest (parent, key, final,
// the new state of a representative), and with RF_CSIZE the sizes of the
// pieces and clusters at their nodes.
struct PottsDev {
    int32_t dim, L, q, flags;          // flags: RF_OPEN | RF_CSIZE | RF_PCC | RF_WIND
    int32_t ntx, nty, ntz, ntiles;     // tiles along x, y, z (1 in 2D)
    int64_t N;
    uint64_t thr, seed;
    uint8_t *spin, *bond;              // N states (read by launch 0, written by the last), N bond bytes
    int32_t *label;                    // N labels of the last sweep
    uint16_t *code;                    // ntiles * sites-per-tile
    uint32_t *cross;                   // ntiles * cross words
    int2 *node;                        // ntiles * slots: {parent, key}
    uint32_t *nfinal;                  // ntiles * slots: a representative's cluster root (last sweep of a call)
    uint8_t *nstate;                   // ntiles * slots: a representative's new state
    uint8_t *kstate;                   // ntiles * slots: the state a representative's piece takes as a cluster's root
    int32_t *psize, *csize;            // ntiles * slots (RF_CSIZE only)
    int4 *wlink;                       // RF_WIND: ntiles * slots node links {parent, dx, dy, dz}
    // PCC (null otherwise): the threshold lives on the device and follows the
    // feedback; per node and axis a < dim, a root's candidate id (cid, id + 2),
    // per border piece its occupied coordinates (pmask), per axis the number of
    // candidates (ncand[a]; ncand[3] counts finished cover blocks), their
    // coverage (cov + a F W, F = L^(dim-1) face sites, W = ceil(L / 32) words per
    // candidate) and how many coordinates each covers (ccount + a F)
    uint64_t *thr_dev;
    uint32_t *pmask;
    int32_t *cid, *ccount, *ncand;
    uint32_t *cov;
};

// Tile counts and per-tile sizes of a Potts lattice's scratch.
struct PottsGeometry {
    int32_t ntx, nty, ntz, ntiles;
    int32_t sites_per_tile, slots, cross_words, pmask_words;
};
__attribute__((visibility("hidden"))) void potts_geometry(int dim, int L, PottsGeometry *g);
__attribute__((visibility("hidden"))) cudaError_t potts_enqueue_hot_start(const PottsDev &p, cudaStream_t st);
// Launch j (0 .. nsweeps) of a call: the tile kernel, then (j < nsweeps) the merge of sweep j.
__attribute__((visibility("hidden"))) cudaError_t potts_enqueue_tile(const PottsDev &p, int j, int nsweeps,
                                                                     uint64_t sweep0, DevObs *obs, cudaStream_t st,
                                                                     bool chained);
__attribute__((visibility("hidden"))) cudaError_t potts_enqueue_merge(const PottsDev &p, int j, int nsweeps,
                                                                      uint64_t sweep0, DevObs *obs, cudaStream_t st,
                                                                      bool chained);
// One call of nsweeps sweeps (observables into obs[0 .. nsweeps-1]).
__attribute__((visibility("hidden"))) cudaError_t potts_enqueue_sweeps(const PottsDev &p, int nsweeps,
                                                                       uint64_t sweep0, DevObs *obs,
                                                                       cudaStream_t st);
__attribute__((visibility("hidden"))) cudaError_t potts_enqueue_check(const uint8_t *s, int64_t n, int q, int32_t *bad,
                                                                      cudaStream_t st);

}  // namespace swg
