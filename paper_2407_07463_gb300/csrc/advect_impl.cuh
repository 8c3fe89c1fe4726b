// Directionally split geometric advection of the active colour fields
// (Section 2.2 transport of every C_i; Section 2.3: one transport equation
// per tracer), per sweep:
//
//   face_flux  one thread per listed face whose upwind donor is interfacial
//              (0 < c < 1): MYC normal and plane constant of the donor, PLIC
//              volume of the swept sub-cell.  Listing keeps the costly
//              reconstruction on full warps.  With a learned normal the FP32
//              path runs face_flux_learned instead (tiles of 128 listed
//              faces through the network on the tensor cores).
//   update     c <- c - (F_hi - F_lo) + c_c (s_hi - s_lo) on the words that
//              can change (boxes.cuh), c_c = [c > 1/2] at the step's start
//              (Weymouth & Yue 2010); empty/full donors give F = 0 / s.  The
//              same pass lists the faces of the NEXT sweep whose donor is
//              interfacial, records c_c as bits in the first sweep, and in
//              the last sweep clips to [0,1] and writes the occupancy bits
//              used by the near-contact test.
//
// Derived quantities (normals, plane constants) never leave the chip.
#pragma once

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "boxes.cuh"
#include "faces.cuh"
#include "plic.cuh"
#include "update_vec.cuh"

namespace vof {

// Buffers and settings shared by the boxes of one advance (internal).
struct SweepArgs {
    unsigned long long* list;    // two face lists of list_entries entries each
    long long list_entries;      // reserved entries per list
    int* counts;                 // [2] their lengths
    long long step;              // index of the first step
    double band;                 // FP64 plane-constant band (FP32 path)
    double tau;                  // occupancy threshold
    bool list_valid;             // list[list_cur] holds the first sweep's faces
    int list_cur;
    cudaStream_t stream;
    long long* launches;
    Prof* prof;
    // learned normal (FP32 path only; null = MYC everywhere)
    const MlpBlob* mlp;
    float mlp_tol;                     // residual at or below which the network is kept outright
    int* mlp_status;                   // set on a timed-out tensor-core wait
    unsigned long long* mlp_counters;  // [0] faces on the network's normal, [1] on MYC's
    int update_blocks_per_sm;          // resident blocks per SM of the update pass (0 = what fits)
};


// Rows of whole 16-byte lanes on 16-byte-aligned buffers take VW cells per
// lane, others (a context only) one.
template <typename T, int NB>
inline bool rows_vectorisable(const BoxSet<T, NB>& S) {
    if (NB > 1) return true;
    const BoxDev<T>& B = S.b[0];
    return B.g.nx % VecOf<T>::W == 0 && (((uintptr_t)B.c | (uintptr_t)B.u) & 15) == 0;
}

// Blocks of a list-writing pass: what the GPU holds at once, the tiles dealt
// out in turn (equal numbers of tiles per block, with fewer blocks, left SMs
// with three blocks beside SMs with four: 5 to 20% of the pass).
template <typename T, int NB>
int sweep_grid(const BoxSet<T, NB>& S, bool vec, const SweepArgs& a) {
    int per_sm = a.update_blocks_per_sm;
    if (per_sm <= 0) per_sm = std::max(1, vec ? update_blocks_per_sm<T, NB, VecOf<T>::W>() : update_blocks_per_sm<T, NB, 1>());
    return std::min(S.tiles, sm_count() * per_sm);
}

// Whether the reserved lists hold every face the set can list.
template <typename T, int NB>
bool lists_fit(const BoxSet<T, NB>& S, const SweepArgs& a) {
    long long need = 0;
    for (int b = 0; b < S.n; ++b) need += list_reserve(S.b[b].words, S.b[b].K);
    return need <= a.list_entries;
}

// Sweep buffers and maps before the first step.
template <typename T, int NB>
cudaError_t clear_set(const BoxSet<T, NB>& S, cudaStream_t st) {
    if (S.tiles <= 0) return cudaSuccess;
    k_clear_sp<T, NB><<<std::min(S.tiles, sm_count() * 8), kSweepThreads, 0, st>>>(S);
    return cudaGetLastError();
}

template <typename T, int NB>
void face_fluxes(const BoxSet<T, NB>& S, int d, int sweep, const unsigned long long* list, const int* count,
                 int* next_count, SweepArgs& a) {
    if constexpr (std::is_same<T, float>::value) {
        if (a.mlp) {
            if (a.prof) a.prof->begin(P_NET_NORMALS);
            face_normals_net_set<NB>(S, d, sweep, list, count, next_count, a.mlp, a.mlp_status, a.stream);
            if (a.prof) { a.prof->end(); a.prof->begin(P_FACE_FLUX); }
            face_flux_judged_set<NB>(S, d, sweep, (float)a.band, list, count, a.mlp_tol, a.mlp_counters, a.stream);
            if (a.prof) a.prof->end();
            if (a.launches) *a.launches += 2;
            return;
        }
    }
    if (a.prof) a.prof->begin(P_FACE_FLUX);
    k_face_flux_bx<T, NB><<<sm_count() * 16, kFaceTile, 0, a.stream>>>(S, d, sweep, (T)a.band, list, count, next_count);
    if (a.prof) a.prof->end();
    if (a.launches) *a.launches += 1;
}

// nsteps steps of every box of S (Section 2.2 split advection with the
// Weymouth & Yue term; c_c bits, clip and occupancy bits as in k_update_sp).
template <typename T, int NB>
cudaError_t advect_set(const BoxSet<T, NB>& S, SweepArgs& a, int nsteps) {
    if (S.n == 0 || nsteps <= 0) return cudaSuccess;
    const bool vec = rows_vectorisable(S);
    const int gb = sweep_grid(S, vec, a);
    if (!lists_fit(S, a)) return cudaErrorInvalidValue;
    unsigned long long* lists[2] = {a.list, a.list + a.list_entries};
    int* counts[2] = {a.counts, a.counts + 1};
    const T tau = (T)a.tau;
    for (int s = 0; s < nsteps; ++s) {
        const long long step = a.step + s;
        const int rot = (int)(step % 3);
        if (!a.list_valid) {
            if (a.prof) a.prof->begin(P_FIND_FACES);
            const cudaError_t z = cudaMemsetAsync(counts[a.list_cur], 0, sizeof(int), a.stream);
            if (z != cudaSuccess) return z;
            launch_list(S, vec, rot, tau, lists[a.list_cur], counts[a.list_cur], gb, a.stream);
            if (a.prof) a.prof->end();
            if (a.launches) *a.launches += 1;
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
        for (int sw = 0; sw < 3; ++sw) {
            const int d = (rot + sw) % 3;
            // next sweep: within the step, or the first sweep of the next step
            const int dn = sw < 2 ? (rot + sw + 1) % 3 : (int)((step + 1) % 3);
            const int cur = a.list_cur, nxt = 1 - a.list_cur;
            // every launch's error is taken where it happens (a later launch's
            // query would clear it)
            face_fluxes(S, d, sw, lists[cur], counts[cur], counts[nxt], a);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            if (a.prof) a.prof->begin(P_UPDATE);
            e = launch_update(S, vec, d, dn, sw, tau, lists[nxt], counts[nxt], gb, a.stream);
            if (e != cudaSuccess) {
                if (a.prof) a.prof->end();
                return e;
            }
            if (a.prof) a.prof->end();
            if (a.launches) *a.launches += 1;
            a.list_cur = nxt;
        }
        a.list_valid = true;
    }
    return cudaGetLastError();
}

// The current face list after Step 4 moved drops of a single box: faces
// whose donor moved change field (k_list_patch); d is the direction of the
// sweep the list serves.  The list geometry is the one advect_set used.
template <typename T>
cudaError_t patch_list_set(const BoxSet<T, 1>& S, SweepArgs& a, int d, const uint32_t* bits, const int* labels,
                           const MoveTables& mt, const int* target) {
    if (!a.list_valid) return cudaSuccess;
    unsigned long long* list = a.list + (a.list_cur ? a.list_entries : 0);
    k_list_patch<T><<<sm_count() * 8, 256, 0, a.stream>>>(S, d, list, a.counts + a.list_cur, bits, labels, mt, target);
    if (a.launches) *a.launches += 1;
    return cudaGetLastError();
}

// Listing from c and the first sweep of step a.step only (c -> first
// scratch buffer; c itself is not modified): a representative, repeatable
// unit of work for timing launch shapes.
template <typename T, int NB>
cudaError_t advect_first_sweep(const BoxSet<T, NB>& S, SweepArgs& a) {
    if (S.n == 0) return cudaSuccess;
    const bool vec = rows_vectorisable(S);
    const int gb = sweep_grid(S, vec, a);
    if (!lists_fit(S, a)) return cudaErrorInvalidValue;
    unsigned long long* lists[2] = {a.list, a.list + a.list_entries};
    int* counts[2] = {a.counts, a.counts + 1};
    const int rot = (int)(a.step % 3), dn = (rot + 1) % 3;
    cudaError_t e = cudaMemsetAsync(counts[0], 0, sizeof(int), a.stream);
    if (e != cudaSuccess) return e;
    launch_list(S, vec, rot, (T)a.tau, lists[0], counts[0], gb, a.stream);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    face_fluxes(S, rot, 0, lists[0], counts[0], counts[1], a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_update(S, vec, rot, dn, 0, (T)a.tau, lists[1], counts[1], gb, a.stream);
}

}  // namespace vof
