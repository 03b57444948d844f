// Declarations of the batched kernels (batch.cu), shared with the host code
// that builds a batch (api.cpp); not part of the ABI.
#pragma once

#include "hs_impl.h"

namespace hs {

// ---- batched persistent kernel (batch.cu)
// One member lattice (periodic sc, stencil layout; every member of a batch in
// one precision, vector width batch_vec(precision)).
struct BatchMember {
    void *planes;           // six planes of the storage type
    int Lx, Ly, Lz, Lh;
    FastDiv div_nxv, div_ly;
    float fJ, fK, fe[3], fbeta;
    double J, K, beta;      // the same in FP64 (FP64 members)
    double e[3];
    const ulonglong2 *sc_tab;  // FP64 members: the trial's sine and cosine table
    float fdelta;              // FP64 members: as PassArgs::fdelta
    int zaxis;              // 1: e = (0, 0, 1) exactly
    uint32_t key0, key1, replica;
    uint32_t sweep0;        // the member's sweep index at batch sweep 0
    double n_present;
    DevAccum *acc;
    int seg_begin, seg_end;  // the member's segments (contiguous)
};

// Items begin, begin + stride, ... (< end) of one member's colour pass,
// each the first of kBlock consecutive items that one CTA's threads take
// together: stride kBlock for a contiguous range; a multiple of kBlock when
// several CTAs sweep one member side by side.
struct BatchSeg {
    int member;
    uint32_t begin, end, stride;
};

struct BatchArgs {
    const BatchMember *members;
    int n_members;
    const BatchSeg *segs;
    const int *cta_seg;      // CTA c owns segments [cta_seg[c], cta_seg[c+1])
    int n_segs;
    double *slots;           // [sweep parity][colour][segment][kPartials]
    unsigned int *bar;       // grid barrier: one 64-bit arrival count (two words, 8-byte aligned)
    int *error;              // latched device error (barrier timeout)
    int n_total, n_equil;    // sweeps, of which the first n_equil unmeasured
    int inject_skip;         // test hook: 1 = CTA 0 skips its first barrier arrival
    int zaxis_all;           // 1: every member's easy axis is (0, 0, 1): FP32 / FP16 run the S.e = S_z kernels
    int kzero_all;           // 1: besides, every member's K is +0: they run the kernels without the K term
    double *group;           // sums of the cluster schedule's sweeps (batch_cluster_bytes)
    const FastDiv *member_rows;  // that schedule: division by each member's Lx / 2 (one site per work item)
};

// sites per work item of a batch member: 16-byte loads for FP64 and FP32,
// 8-byte loads for FP16
inline int batch_vec(int precision) { return precision == HS_FP64 ? 2 : 4; }
// prefetch 0: one work item of loads at a time; 1: split prefetch (the
// next item's DRAM-heavy rows load during the current item's arithmetic)
cudaError_t launch_batch(int precision, const BatchArgs &b, int grid, cudaStream_t s, int prefetch);
// the per-pass schedule: 2 n_total chained pass launches and a finalise launch
cudaError_t launch_batch_passes(int precision, const BatchArgs &b, int grid, cudaStream_t s, int prefetch);
int batch_occupancy(int precision, int prefetch);
// the resident schedule: one CTA per member, its planes in dynamic shared
// memory (smem bytes, at most batch_resident_limit(precision)) for the whole run
cudaError_t launch_batch_resident(int precision, const BatchArgs &b, size_t smem, cudaStream_t s);
size_t batch_resident_limit(int precision);
// the resident schedule of FP64 batches of few members: one cluster of ctas
// CTAs (0: none) of that many threads per member, for members of at most
// kBatchClusterSites sites: us per sweep in clusters and on the persistent
// schedule, of 12, 24, 48 and 76 members of 24^3 (13,824 sites) 20.2 and 30.6, 27.1
// and 35.5, 52.5 and 55.5, 52.4 and 69.7; of 16,384 sites 20.5 and 28.8, 32.3 and
// 39.1, 63.0 and 58.5, 58.7 and 71.9; of 24,576 27.0 and 31.0, 39.8 and 45.9, 77.7 and
// 72.3, 83.6 and 94.6; of 32^3 32.7 and 40.9, 51.4 and 57.6, 101 and 84, 109 and 117
constexpr int64_t kBatchClusterSites = 16384;
struct BatchClusters {
    int ctas, threads;
};
BatchClusters batch_cluster_plan(int precision, int n_members, int64_t max_sites, int n_sm);
size_t batch_cluster_bytes(int n_members, const BatchClusters &p);
cudaError_t launch_batch_clusters(const BatchArgs &b, const BatchClusters &p, cudaStream_t s);
// zero every member's accepted-move counter (reads b.members on the device)
cudaError_t launch_batch_reset(const BatchArgs &b, cudaStream_t s);

}  // namespace hs
