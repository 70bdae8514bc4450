// expand_internal.h -- device layout of a frontier (the evaluated set V and
// the next batch) shared by expand.cu and frontier.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "comet.h"

namespace comet {

constexpr int kTopMax = 4096;         // the largest k of a top-k
constexpr int kRun = 256;             // keys of a run ranked by counting
constexpr int kMerge = 8;             // runs merged at a time
constexpr int kScan = 1024;           // slots per block of the compaction
constexpr int kMaxGridY = 65535;      // frontiers per launch

struct alignas(16) TopKey {
    uint32_t mk;    // order-preserving key of M_hat
    uint32_t idx;   // position of the entry in the ranked array (first pass)
    uint64_t code;  // mode code (tie break)
};

// Keys that the top-k passes over up to n keys write into top_a (pass 0, and
// every other one) and top_b, for k up to k_max; callers copy k keys of either.
inline int64_t top_a_keys(int64_t n, int k_max) {
    return std::max<int64_t>((n + kRun - 1) / kRun * std::min(k_max, kRun), kTopMax);
}
inline int64_t top_b_keys(int64_t n, int k_max) {
    const int64_t runs = (n + kRun - 1) / kRun;
    return std::max<int64_t>((runs + kMerge - 1) / kMerge * std::min(k_max, kMerge * kRun), kTopMax);
}

struct FrontierDev {
    int instance, n_modes, lmax, slots;
    // neighbourhood rule: edit radius (1, 2), grammar (0 = every order over
    // the instance's modes; 1 = the pushing grammar over stick-on-a-face and
    // free motion), alphabet size and one-edit slots per order
    int radius, grammar, n_alpha, slots1;
    int64_t capacity;     // |V| maximum
    int64_t batch_cap;    // largest batch added at once
    unsigned long long* codes;  // [capacity]
    float* merit;               // [capacity]
    unsigned long long* nV;     // |V|
    unsigned long long* set;    // hash set of V's codes
    unsigned long long set_mask;
    TopKey* top_a;              // top-k pass buffers
    TopKey* top_b;
    unsigned long long* cand_code;  // [k_max * slots] proposed codes, then the winners'
    int* flag;                      // [k_max * slots] entry of a proposal in the candidate table
    int* counts;                    // winners per kScan slots
    unsigned long long* cand_keys;  // candidate table, empty (zero) between rounds
    unsigned int* cand_ord;
    unsigned long long cand_mask;
    int batch;                      // orders of the next batch
    comet_mode_seq* next;           // [batch]
    int64_t* n_next;
    int* error;                     // 1 malformed order, 2 capacity exceeded
};

// one-edit slots of an order under a rule (fixed layout over l_max:
// substitutions l_max x n_alpha, insertions (l_max + 1) x n_alpha, deletions
// l_max) and all slots per parent (radius 2 adds slots1 x slots1)
inline int64_t edit_slots1(int lmax, int n_alpha) { return (int64_t)lmax * n_alpha * 2 + n_alpha + lmax; }
inline int64_t edit_slots(int lmax, int n_alpha, int radius) {
    const int64_t s1 = edit_slots1(lmax, n_alpha);
    return radius == 2 ? s1 + s1 * s1 : s1;
}
constexpr int kGrammarNone = 0, kGrammarPush = 1;
constexpr int kPushFree = 12;  // free motion in the 13-mode pushing alphabet

cudaError_t launch_frontier_restore(const FrontierDev& F, int64_t n, cudaStream_t s);
cudaError_t launch_frontier_add(const FrontierDev& F, const comet_mode_seq* seqs, int64_t n, const int64_t* d_n,
                                const float* cost, const float* viol, float eps_feas, float merit_mu, cudaStream_t s);
const TopKey* launch_topk(const FrontierDev& F, int k, cudaStream_t s, cudaError_t* err);
cudaError_t launch_expand(const FrontierDev& F, int k, int batch, int64_t budget, cudaStream_t s);
// the same for n_f frontiers (an array in device memory) in one launch each
cudaError_t launch_frontier_add_many(const FrontierDev* d_fs, int n_f, const comet_mode_seq* seqs, const int64_t* d_off,
                                     bool seeds, int64_t n_max, const float* cost, const float* viol, float eps_feas,
                                     float merit_mu, cudaStream_t s);
cudaError_t launch_topk_many(const FrontierDev* d_fs, int n_f, int64_t capacity, int k, bool* in_b, cudaStream_t s);
cudaError_t launch_expand_many(const FrontierDev* d_fs, int n_f, int64_t capacity, int64_t slots, int k,
                               int64_t budget, cudaStream_t s);

}  // namespace comet

struct comet_problem;

struct comet_frontier {
    comet_problem* p = nullptr;
    comet::FrontierDev d;
    int32_t batch = 0;
    int32_t k_max = 0;
    void* blob = nullptr;  // one allocation for all device arrays
};
