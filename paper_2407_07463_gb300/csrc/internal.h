// Internal host-side launchers of the GB300 VoF library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

#include <vector>

namespace vof {

// Kernel classes of the launch timer (vof_profile_*).
enum ProfClass {
    P_FIND_FACES = 0,
    P_FACE_FLUX,
    P_UPDATE,
    P_PACK_BITS,
    P_NEAR_CONTACT,
    P_LABEL,
    P_PAIRS,
    P_TOUCH,
    P_MOVE,
    P_STATS,
    P_MISC,
    P_NET_NORMALS,
    P_COUNT
};

// Optional CUDA-event bracketing of kernel launches on one stream.
struct Prof {
    bool on = false;
    int cap = 0, n = 0, pending = -1;
    std::vector<cudaEvent_t> ev;  // 2 * cap
    std::vector<int> cls;         // cap
    cudaStream_t st = nullptr;
    void begin(int c) {
        pending = -1;
        if (!on || n >= cap) return;
        cudaEventRecord(ev[2 * n], st);
        pending = c;
    }
    void end() {
        if (pending < 0) return;
        cudaEventRecord(ev[2 * n + 1], st);
        cls[n] = pending;
        ++n;
        pending = -1;
    }
};

constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kPairCap = 1 << 16;     // distinct tagged near-contact pairs per call
constexpr int kMoveCap = 2048;        // moving drops per recolour call
constexpr int kDropCap = 1 << 20;     // drops over all fields for statistics

// Keeps the name of the last CUDA error a library call met (for
// vof_last_cuda_error); returns the error unchanged.
cudaError_t note_cuda_error(cudaError_t e);
const char* last_cuda_error_name();
struct SweepArgs;
struct MlpBlob;
struct MoveTables;
template <typename T, int NB>
struct BoxSet;
constexpr int kMaxBoxes = 64;
// Learned normal of a box set (FP32 path): network normals of the listed
// faces of one sweep (tensor cores; *next_count, the count of the list that
// the sweep's update pass will fill, set to zero), then their judged fluxes;
// counters[0/1] += faces on the network's / MYC's normal.
template <int NB>
void face_normals_net_set(const BoxSet<float, NB>& S, int d, int sweep, const unsigned long long* list,
                          const int* count, int* next_count, const MlpBlob* w, int* status, cudaStream_t st);
template <int NB>
void face_flux_judged_set(const BoxSet<float, NB>& S, int d, int sweep, float band, const unsigned long long* list,
                          const int* count, float tol, unsigned long long* counters, cudaStream_t st);
// nsteps steps of every box of a set (one box: a context; up to kMaxBoxes:
// a batch).
cudaError_t advect_set_fp64(const BoxSet<double, 1>& S, SweepArgs& a, int nsteps);
cudaError_t advect_set_fp32(const BoxSet<float, 1>& S, SweepArgs& a, int nsteps);
cudaError_t advect_set_fp64(const BoxSet<double, kMaxBoxes>& S, SweepArgs& a, int nsteps);
cudaError_t advect_set_fp32(const BoxSet<float, kMaxBoxes>& S, SweepArgs& a, int nsteps);
// After Step 4 moved drops of a context's box: the faces of the current
// list whose donor moved take the drop's target field (d: the direction of
// the sweep the list serves; bits and labels: Step 1's occupancy and Step
// 2's tags; target[m]: the field drop m moved to, or -1).
cudaError_t patch_list_fp32(const BoxSet<float, 1>& S, SweepArgs& a, int d, const uint32_t* bits, const int* labels,
                            const MoveTables& mt, const int* target);
cudaError_t patch_list_fp64(const BoxSet<double, 1>& S, SweepArgs& a, int d, const uint32_t* bits, const int* labels,
                            const MoveTables& mt, const int* target);
// Resident blocks per SM of a batch's update pass (0 if the query fails),
// asked of the unit that launches it.
int update_occupancy(bool fp64);
int update_occupancy_fp64();
// Sweep buffers (the active fields) and their maps before the first step of a set.
cudaError_t clear_set_fp64(const BoxSet<double, 1>& S, cudaStream_t st);
cudaError_t clear_set_fp32(const BoxSet<float, 1>& S, cudaStream_t st);
cudaError_t clear_set_fp64(const BoxSet<double, kMaxBoxes>& S, cudaStream_t st);
cudaError_t clear_set_fp32(const BoxSet<float, kMaxBoxes>& S, cudaStream_t st);
// Listing and first sweep of a batch only (state untouched; for timing).
cudaError_t advect_first_sweep_fp64(const BoxSet<double, kMaxBoxes>& S, SweepArgs& a);
cudaError_t advect_first_sweep_fp32(const BoxSet<float, kMaxBoxes>& S, SweepArgs& a);
// Face-list entries to reserve per list for K fields of `words` 32-cell
// words: up to 2 faces per cell.
inline long long list_reserve(long long words, int K) { return 64LL * K * words; }

// Face lists: consumers take tiles of kFaceTile consecutive entries.
constexpr int kFaceTile = 128;
cudaError_t pack_bits(const void* c, bool fp64, uint32_t* bits, const Dims& g, int K, double tau,
                      cudaStream_t st);
// Box dilation (Chebyshev distance reach, periodic) of n bit planes from src
// into dst; tmp: n planes of scratch.
cudaError_t dilate_planes(const uint32_t* src, uint32_t* dst, uint32_t* tmp, int n, const Dims& g, int reach,
                          cudaStream_t st);
// Step 1 per field: flags[f] |= 1 if it fired, |= 2 if the field holds an
// occupied cell (flags cleared by the caller).
cudaError_t near_contact(const uint32_t* bits, uint32_t* ncmap, int* flags, const Dims& g, int K, int w,
                         cudaStream_t st);
// Tags of one field's occupancy bits: label (0 empty, else 1 + the rank of
// the component's root, its smallest cell), *n_out the tag count, root_of[l
// - 1] the root cell of tag l <= root_cap (if not null).  parent, rank,
// block_tot and block_off are scratch: parent does not hold every cell's
// root afterwards.
cudaError_t label_field(const uint32_t* bits_f, const Dims& g, int conn, int* parent, int* rank,
                        int* block_tot, int* block_off, int* label, int* root_of, int root_cap, int* n_out,
                        cudaStream_t st, long long* launches);
// Fields tagged by one chain of launches (slot s = blockIdx.y takes field
// f[s]).  A field's bit plane, near-contact map and labels sit f * words and
// f * N from their bases and its drop count at n_out[f]; a slot's scratch
// sits s * N (parent, rank) and s * (nb + 1) (block totals and offsets, nb =
// ceil(N / 1024)) from theirs.  Labels are complete only at occupied cells
// (empty cells of a row word without an occupied cell keep what they held).
// root_of (not null): the tags' root cells, slot after slot.
constexpr int kLabelSlots = 16;
struct LabelSlots {
    int n;
    int f[kLabelSlots];
};
cudaError_t label_fields(const uint32_t* bits, const Dims& g, int conn, const LabelSlots& ls, int* parent, int* rank,
                         int* block_tot, int* block_off, int* labels, int* n_out, cudaStream_t st,
                         long long* launches, int* root_of = nullptr, int root_cap = 0);
// Step 3 for the slots' fields: distinct pairs of the tags of opposite
// occupied cells around every near-contact cell, into the set `table`.
cudaError_t tag_pairs_fields(const uint32_t* ncmap, const uint32_t* bits, const int* labels, const Dims& g, int w,
                             const LabelSlots& ls, unsigned long long* table, int cap, int* overflow,
                             cudaStream_t st);
cudaError_t compact_pairs(const unsigned long long* table, int cap, unsigned long long* out,
                          unsigned long long* count, cudaStream_t st);

// Step 4 helpers.  Moving drops are listed per field in increasing label
// order: mv_label[mv_start[f] .. mv_start[f] + mv_count[f]).
// mv_map: a bit per (field, tag) below kMoveMapTags, set for moving drops
// (a lookup without the search); larger tags are searched.
constexpr int kMoveMapTags = 1 << 16;
constexpr int kMoveMapWords = kMoveMapTags / 32;  // per field
struct MoveTables {
    const int* mv_start;      // [K]
    const int* mv_count;      // [K]
    const int* mv_label;      // [M]
    int M;
    const uint32_t* mv_map;   // [K][kMoveMapWords]
};

#ifdef __CUDACC__
// Index of label l among field f's moving drops, or -1.
__device__ __forceinline__ int moving_index(const MoveTables& mt, int f, int l) {
    int lo = mt.mv_start[f], n = mt.mv_count[f];
    int a = 0, b = n - 1;
    while (a <= b) {
        int mid = (a + b) >> 1;
        int v = mt.mv_label[lo + mid];
        if (v == l) return lo + mid;
        if (v < l) a = mid + 1;
        else b = mid - 1;
    }
    return -1;
}

// Is tag l (> 0) of field f a moving drop?
__device__ __forceinline__ bool is_moving(const MoveTables& mt, int f, int l) {
    if (l <= 0) return false;
    if (l < kMoveMapTags) return (mt.mv_map[(size_t)f * kMoveMapWords + (l >> 5)] >> (l & 31)) & 1u;
    return moving_index(mt, f, l) >= 0;
}
#endif
// Moving-drop bits (mvbits: a plane per field of mv_fields), then touch[m]
// and conflict[m] for every moving drop; dil: scratch of n_active +
// 2 n_mv_fields bit planes; reach <= 16, n_active and n_mv_fields <= 32.
cudaError_t recolour_touch(const int* labels, const uint32_t* bits, uint32_t* mvbits, uint32_t* dil, const Dims& g,
                           int n_active, int reach, MoveTables mt, const int* mv_fields, int n_mv_fields,
                           unsigned* touch, unsigned* conflict, int Mw, cudaStream_t st, long long* launches);
// The bit map of moving tags (mt.mv_map, cleared by the caller) for the
// n_fields fields listed in mv_fields.
cudaError_t move_map(MoveTables mt, uint32_t* map, const int* mv_fields, int n_fields, cudaStream_t st);
// Moves the cells set in mvbits to their drop's target field, whose bits of
// the maps of non-zero words (nzc, 16 bits per word) and end cells (nze, twice
// 16 bits) are set.
cudaError_t recolour_move(void* c, bool fp64, const int* labels, const uint32_t* mvbits, const Dims& g,
                          MoveTables mt, const int* mv_fields, int n_mv_fields, const int* target, uint16_t* nzc,
                          uint32_t* nze, cudaStream_t st);

// Statistics helpers.
// Drops of the slots' fields, counted slot after slot (a single field: one
// slot with f[0] = 0 and its own pointers).  c and labels: the fields f * N
// from their bases; bits (may be null): occupancy the labels were made from
// (words without an occupied cell are skipped unread), else every label is
// read; n_out[f]: tags of field f (null with one slot); n_max: most drops.
struct DropFields {
    const void* c;
    bool fp64;
    const int* labels;
    const uint32_t* bits;
    const int* n_out;
    LabelSlots ls;
    int n_max;
};
// Smallest cell of every tag (root_of[0 .. n_max)).
cudaError_t drop_roots(const DropFields& D, const Dims& g, int* root_of, cudaStream_t st);
// Per drop: the sum of c and its first moments about its root cell (minimum
// image), into S[4 drop ..] (cleared first).
cudaError_t drop_sums(const DropFields& D, const Dims& g, const int* root_of, double* S, cudaStream_t st);
cudaError_t drop_finalize(const double* S, const int* root_of, const Dims& g, double h, int n,
                          double* vol, double* cen, cudaStream_t st);
// Height-function curvatures of K fields (NaN where an interfacial cell has
// none; with fill also in every other cell, which is otherwise not written)
// and the surface-tension source f[3][N] = sum over K fields of gamma kappa
// grad c on the low faces (Section 2.3), from curvatures of either kind.
cudaError_t curvature_fields(bool fp64, const void* c, int K, const Dims& g, double h, void* kappa, bool fill,
                             cudaStream_t st);
cudaError_t surface_tension(bool fp64, const void* c, const void* kappa, int K, const Dims& g, double h,
                            double gamma, void* f, cudaStream_t st);
// Drop shape (Appendix A): I[n][6] = xx yy zz xy xz yz about cen (cleared
// first), then chi = sqrt(I_max / I_min) per drop (chi may be null) with
// acc[0] += sum chi, acc[1] += drops, acc[2] = max(acc[2], chi) (acc may be
// null).
cudaError_t drop_inertia(const DropFields& D, const Dims& g, double h, const double* cen, double* I, cudaStream_t st);
cudaError_t drop_chi(const double* I, int n, double* chi, double* acc, cudaStream_t st);
cudaError_t pair_stats(const double* cen, long long n, double bx, double by, double bz, int vaxis,
                       int n_rbins, double dr, int n_tbins, double dtheta, double tie_tol, double* hist_r,
                       double* hist_rt, double* moments, cudaStream_t st);

// Learned normal estimator.
struct MlpBlob;
cudaError_t mlp_forward(const MlpBlob* w, const float* st, float* n_out, long long n, int* status,
                        cudaStream_t stream);
cudaError_t mlp_grad_pass(const MlpBlob* w, const float* st, const float* tgt, long long n0, long long n,
                          float inv_batch, float* grad, float* loss_sum, int* status, cudaStream_t stream);
cudaError_t tc_gemm_check(const float* A, const float* B, float* D, int K, int N, int swap, int* status,
                          cudaStream_t st);

// PLIC primitives and normals (tests and tools).
cudaError_t plic_volume_batch(bool fp64, const void* m, const void* alpha, void* v, long long n,
                              cudaStream_t st);
cudaError_t plic_alpha_batch(bool fp64, const void* m, const void* c, void* alpha, long long n,
                             double band, cudaStream_t st);
cudaError_t normals_field(bool fp64, const void* cf, const Dims& g, void* m, cudaStream_t st);
cudaError_t velocity_scan(bool fp64, const void* u, long long n, double* out2, cudaStream_t st);

}  // namespace vof
