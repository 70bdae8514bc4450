// expand.cu -- device side of the greedy local mode expansion (Sec. III-B,
// Algorithm 1): the evaluated set V as a code list plus an open-addressing
// hash set, top-k of V by (M_hat, code), one-edit neighbourhoods of the top
// k in enumeration order, deduplication against V and within the round, and
// compaction of the first B unseen orders into the next batch F_{s+1}.
//
// Every count lives in device memory and every launch has a fixed grid, so
// a whole expansion round can be captured in a CUDA graph.  A launch serves
// one frontier or several at once (blockIdx.y), as the batched planner does.

#include <cuda_runtime.h>
#include <stdint.h>

#include "comet.h"
#include "comet_internal.h"
#include "expand_internal.h"
#include "launch.h"

namespace comet {
namespace {

constexpr unsigned long long kEmpty = 0ull;  // code 0 is never a valid order (length >= 1)

__device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
    // SplitMix64 finaliser (Steele, Lea and Flood 2014) as the hash
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x;
}

// order-preserving map of a float to an unsigned key (NaN -> largest)
__device__ __forceinline__ uint32_t float_key(float f) {
    if (f != f) return 0xffffffffu;
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ unsigned long long encode_seq(const comet_mode_seq& s, int n_modes) {
    const unsigned long long base = (unsigned long long)(n_modes + 1);
    unsigned long long code = s.len, p = base;
    for (int i = 0; i < s.len; ++i) {
        code += (unsigned long long)(s.modes[i] + 1) * p;
        p *= base;
    }
    return code;
}

__device__ int decode_code(unsigned long long code, int n_modes, uint16_t* modes) {
    const unsigned long long base = (unsigned long long)(n_modes + 1);
    const int L = (int)(code % base);
    code /= base;
    for (int i = 0; i < L; ++i) {
        modes[i] = (uint16_t)(code % base - 1);
        code /= base;
    }
    return L;
}

// insert; returns true if the code was not present
__device__ bool set_insert(unsigned long long* set, unsigned long long mask, unsigned long long code) {
    unsigned long long h = mix64(code) & mask;
    for (unsigned long long probe = 0; probe <= mask; ++probe) {
        const unsigned long long prev = atomicCAS(&set[h], kEmpty, code);
        if (prev == kEmpty) return true;
        if (prev == code) return false;
        h = (h + 1) & mask;
    }
    return false;  // table full (capacity is twice the maximum count, so unreachable)
}

__device__ bool set_contains(const unsigned long long* set, unsigned long long mask, unsigned long long code) {
    unsigned long long h = mix64(code) & mask;
    for (unsigned long long probe = 0; probe <= mask; ++probe) {
        const unsigned long long v = set[h];
        if (v == code) return true;
        if (v == kEmpty) return false;
        h = (h + 1) & mask;
    }
    return false;
}

// candidate table: code -> smallest ordinal proposing it.  Ordinals are kept
// inverted (~ord, the largest wins), so that zeroed memory is an empty table;
// each round's winners clear their entries again.  Returns the entry.
__device__ int cand_insert(unsigned long long* keys, unsigned int* ords, unsigned long long mask,
                           unsigned long long code, unsigned int ord) {
    unsigned long long h = mix64(code) & mask;
    for (unsigned long long probe = 0; probe <= mask; ++probe) {
        const unsigned long long prev = atomicCAS(&keys[h], kEmpty, code);
        if (prev == kEmpty || prev == code) {
            atomicMax(&ords[h], ~ord);
            return (int)h;
        }
        h = (h + 1) & mask;
    }
    return -1;  // table full (it holds twice the proposals, so unreachable)
}

// ------------------------------------------------------------- add to V

__device__ void add_orders(const FrontierDev& F, const comet_mode_seq* seqs, int64_t nn, const float* cost,
                           const float* viol, float eps_feas, float merit_mu) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nn; i += (int64_t)gridDim.x * blockDim.x) {
        const comet_mode_seq s = seqs[i];
        if (s.instance != F.instance || s.len < 1 || s.len > F.lmax) {
            atomicExch(F.error, 1);
            continue;
        }
        const unsigned long long code = encode_seq(s, F.n_modes);
        if (!set_insert(F.set, F.set_mask, code)) continue;  // already evaluated
        const unsigned long long slot = atomicAdd(F.nV, 1ull);
        if (slot >= (unsigned long long)F.capacity) {
            atomicExch(F.error, 2);
            continue;
        }
        const float c = cost[i], v = viol[i];
        // Eq. search_merit; a non-finite score ranks last
        float m = c + merit_mu * fmaxf(v - eps_feas, 0.f);
        if (!(m == m) || isinf(m)) m = __int_as_float(0x7f800000);
        F.codes[slot] = code;
        F.merit[slot] = m;
    }
}

__global__ void add_kernel(FrontierDev F, const comet_mode_seq* seqs, int64_t n, const int64_t* d_n, const float* cost,
                           const float* viol, float eps_feas, float merit_mu) {
    add_orders(F, seqs, d_n ? *d_n : n, cost, viol, eps_feas, merit_mu);
}

// frontier y adds its slots [off[y], off[y] + n): n = its own next count, or
// off[y + 1] - off[y] when `seeds`
__global__ void add_many_kernel(const FrontierDev* Fs, const comet_mode_seq* seqs, const int64_t* off, int seeds,
                                const float* cost, const float* viol, float eps_feas, float merit_mu) {
    const FrontierDev F = Fs[blockIdx.y];
    const int64_t o = off[blockIdx.y], n = seeds ? off[blockIdx.y + 1] - o : *F.n_next;
    add_orders(F, seqs + o, n, cost + o, viol + o, eps_feas, merit_mu);
}

// ---------------------------------------------------------------- top-k
// The k smallest keys of V, in order.  Pass 0 ranks every run of kRun keys by
// counting: a key's place is the number of smaller keys in its run (read as
// shared-memory broadcasts), and the first min(k, kRun) stay.  Each later pass
// merges kMerge sorted runs: a key's place is its own plus, by binary search,
// the number of smaller keys in each of the others; the first k stay.  Keys
// are unique in practice; equal ones keep their input order.
//
// Counting needs no barriers and spreads over all SMs, but costs n times the
// run; searching costs n log(run).  So runs are short and the rest is merged.
// Before, every pass counted in chunks of max(4096, 4 k) keys, in one chunk up
// to 16,384; before that, chunks of 4,096 were sorted in a CTA each (78
// barriers, 80 us however small the set).  A comet_frontier_best call, which
// copies k keys back and waits (us: sorted chunks / counted chunks / now):
//      n = 8,000  k = 64     249 /   65 /  45    k = 2,048   254 /   67 /  57
//         20,736             249 /   69 /  55                480 /  127 /  76
//        105,000             251 /  164 /  58                699 /  403 / 101
//        420,000             357 /  537 /  86                921 / 1329 / 197
//      1,048,576             454 / 1321 / 135               1131 / 3173 / 385
// Runs of 128 keys and merges of 8 are as good; runs of 512 take 49 us at 8,000
// keys and 108 at 420,000 (k = 64), merges of 16 more everywhere.
struct Runs {
    int64_t n;      // sorted runs, one after the other
    int len, tail;  // length of every run but the last, and of the last
};

// the runs that pass `pass` >= 1 finds
__device__ Runs runs_at(int64_t n_keys, int pass, int k) {
    Runs R;
    R.n = (n_keys + kRun - 1) / kRun;
    R.len = min(k, kRun);
    R.tail = (int)min((int64_t)k, n_keys - (R.n - 1) * kRun);
    for (int p = 1; p < pass; ++p) {
        const int64_t m = (R.n + kMerge - 1) / kMerge;
        const int64_t last = (R.n - (m - 1) * kMerge - 1) * R.len + R.tail;
        R.n = m;
        R.len = min(k, kMerge * R.len);
        R.tail = (int)min((int64_t)k, last);
    }
    return R;
}

// whether o comes before me; `ties`: also if they are equal (no branches)
__device__ __forceinline__ bool key_before(const TopKey& o, const TopKey& me, bool ties) {
    return (o.mk < me.mk) | ((o.mk == me.mk) & ((o.code < me.code) | (ties & (o.code == me.code))));
}

// |V| may have run past the capacity (flagged on add): never read beyond it
__device__ __forceinline__ int64_t keys_of(const FrontierDev& F) {
    return (int64_t)min(*F.nV, (unsigned long long)F.capacity);
}

__global__ void __launch_bounds__(kRun) topk_rank_kernel(FrontierDev F0, const FrontierDev* Fs, int k) {
    launch_next();
    await_previous();
    // merit keys apart from the codes: four a load, and codes only for a tie
    __shared__ __align__(16) uint32_t mk[kRun];
    __shared__ unsigned long long code[kRun];
    const FrontierDev F = Fs ? Fs[blockIdx.y] : F0;
    const int64_t base = (int64_t)blockIdx.x * kRun;
    const int len = (int)min((int64_t)kRun, keys_of(F) - base), i = threadIdx.x;
    if (len <= 0) return;
    TopKey me;
    me.mk = 0xffffffffu;  // past the end: before no key
    me.idx = (uint32_t)(base + i);
    me.code = ~0ull;
    if (i < len) {
        me.mk = float_key(F.merit[base + i]);
        me.code = F.codes[base + i];
    }
    mk[i] = me.mk;
    code[i] = me.code;
    __syncthreads();
    if (i >= len) return;
    int rank = 0, same = 0;
#pragma unroll 8
    for (int j = 0; j < kRun; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(mk + j);
        rank += (o.x < me.mk) + (o.y < me.mk) + (o.z < me.mk) + (o.w < me.mk);
        same += (o.x == me.mk) + (o.y == me.mk) + (o.z == me.mk) + (o.w == me.mk);
    }
    if (same > 1)
        for (int j = 0; j < len; ++j)
            rank += mk[j] == me.mk && (code[j] < me.code || (code[j] == me.code && j < i));
    if (rank < k) F.top_a[blockIdx.x * (int64_t)min(k, kRun) + rank] = me;
}

// pass 1 reads top_a and writes top_b, pass 2 the other way round, ...
__global__ void __launch_bounds__(256) topk_merge_kernel(FrontierDev F0, const FrontierDev* Fs, int pass, int k) {
    launch_next();
    await_previous();
    const FrontierDev F = Fs ? Fs[blockIdx.y] : F0;
    const TopKey* in = (pass & 1) ? F.top_a : F.top_b;
    TopKey* out = (pass & 1) ? F.top_b : F.top_a;
    const Runs R = runs_at(keys_of(F), pass, k);
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (R.n == 0 || t >= (R.n - 1) * R.len + R.tail) return;
    const int64_t run = t / R.len, group = run / kMerge;
    const TopKey me = in[t];
    // A search is a chain of dependent loads, so all runs of the group are
    // searched side by side, without branches: a step past a run's end (its own
    // run counts as empty) looks at the key itself, which is not before it
    int at[kMerge] = {}, n[kMerge];
#pragma unroll
    for (int u = 0; u < kMerge; ++u) {
        const int64_t j = group * kMerge + u;
        n[u] = j >= R.n || j == run ? 0 : j == R.n - 1 ? R.tail : R.len;
    }
    const TopKey* first = in + group * kMerge * R.len;
    const int own = (int)(run - group * kMerge);
    for (int step = 1 << (31 - __clz(R.len)); step > 0; step >>= 1) {
        TopKey o[kMerge];
#pragma unroll
        for (int u = 0; u < kMerge; ++u)
            o[u] = *(at[u] + step <= n[u] ? first + (int64_t)u * R.len + at[u] + step - 1 : in + t);
#pragma unroll
        for (int u = 0; u < kMerge; ++u)
            if ((at[u] + step <= n[u]) & key_before(o[u], me, u < own)) at[u] += step;
    }
    int64_t rank = t - run * R.len;
#pragma unroll
    for (int u = 0; u < kMerge; ++u) rank += at[u];
    if (rank < k) out[group * min(k, kMerge * R.len) + rank] = me;
}

// --------------------------------------------------------- neighbourhood


// Mode of alphabet position a: every mode (grammar 0), or for the pushing
// grammar stick on face a (mode 3 a, a < 4) and free motion (a = 4).
__device__ __forceinline__ int alpha_mode(const FrontierDev& F, int a) {
    return F.grammar == kGrammarPush ? (a < 4 ? 3 * a : kPushFree) : a;
}

// Pushing grammar (Sec. III-A; the reading fixed by the paper's printed
// counts): the order starts in free motion, no two consecutive segments
// share a mode, every mode is stick-on-a-face or free, and a direct
// contact-to-contact switch joins adjacent faces of the cyclic face list.
__device__ bool admissible(const FrontierDev& F, const uint16_t* s, int L) {
    if (F.grammar != kGrammarPush) return true;
    if (L < 1 || s[0] != kPushFree) return false;
    for (int i = 0; i < L; ++i)
        if (s[i] != kPushFree && (s[i] % 3 != 0 || s[i] >= 12)) return false;
    for (int i = 0; i + 1 < L; ++i) {
        const int a = s[i], b = s[i + 1];
        if (a == b) return false;
        if (a != kPushFree && b != kPushFree) {
            const int d = (a / 3 - b / 3 + 4) & 3;
            if (d != 1 && d != 3) return false;
        }
    }
    return true;
}

// One-edit neighbour of seq (length L) at slot j of the fixed layout:
// substitutions (position < l_max, alphabet position; the current mode is
// skipped), insertions (position <= l_max, alphabet position), deletions
// (position < l_max).  Slots that do not apply to this L are empty.  Within
// an order the slots run in the enumeration order of the neighbourhood.
// Returns the new length, or 0 for an empty slot.
__device__ int neighbour(const FrontierDev& F, const uint16_t* s, int L, int j, uint16_t* out) {
    const int nA = F.n_alpha, lmax = F.lmax;
    if (j < lmax * nA) {
        const int pos = j / nA, m = alpha_mode(F, j % nA);
        if (pos >= L || m == s[pos]) return 0;
        for (int i = 0; i < L; ++i) out[i] = s[i];
        out[pos] = (uint16_t)m;
        return L;
    }
    j -= lmax * nA;
    if (j < (lmax + 1) * nA) {
        const int pos = j / nA, m = alpha_mode(F, j % nA);
        if (L + 1 > lmax || pos > L) return 0;
        for (int i = 0, o = 0; i <= L; ++i) {
            if (i == pos) out[o++] = (uint16_t)m;
            if (i < L) out[o++] = s[i];
        }
        return L + 1;
    }
    j -= (lmax + 1) * nA;
    if (j < lmax && L - 1 >= 1 && j < L) {
        for (int i = 0, o = 0; i < L; ++i)
            if (i != j) out[o++] = s[i];
        return L - 1;
    }
    return 0;
}

// N_r(m) slot j (Sec. III-B): j < slots1 is a one-edit neighbour; with
// radius 2, j = slots1 + j1 slots1 + j2 is neighbour j2 of neighbour j1 (so
// the one-edit orders come first, then the two-edit ones grouped by their
// intermediate).  Every order on the way must be admissible; the parent
// itself is not a neighbour.  Returns the length, or 0.
__device__ int neighbour_r(const FrontierDev& F, const uint16_t* s, int L, int j, uint16_t* out) {
    if (j < F.slots1) {
        const int Ln = neighbour(F, s, L, j, out);
        return (Ln > 0 && admissible(F, out, Ln)) ? Ln : 0;
    }
    j -= F.slots1;
    uint16_t mid[COMET_MAX_SEGMENTS];
    const int Lm = neighbour(F, s, L, j / F.slots1, mid);
    if (Lm == 0 || !admissible(F, mid, Lm)) return 0;
    const int Ln = neighbour(F, mid, Lm, j % F.slots1, out);
    if (Ln == 0 || !admissible(F, out, Ln)) return 0;
    if (Ln == L) {
        bool same = true;
        for (int i = 0; i < L; ++i) same = same && out[i] == s[i];
        if (same) return 0;
    }
    return Ln;
}

// One thread per edit slot; a slot that proposes an unseen order leaves its
// code and its entry in the candidate table.  A block's slots belong to a few
// consecutive parents, whose codes are decoded once per block: a decode is up
// to 16 dependent 64-bit divisions, most of a slot's work otherwise (35 us
// against 26 us for the 560,000 slots of a two-edit round).
constexpr int kNbThreads = 256;

__global__ void __launch_bounds__(kNbThreads) neighbour_kernel(FrontierDev F0, const FrontierDev* Fs, int in_b, int k) {
    launch_next();
    await_previous();
    __shared__ uint16_t par[kNbThreads][COMET_MAX_SEGMENTS];
    __shared__ int par_len[kNbThreads];
    const FrontierDev F = Fs ? Fs[blockIdx.y] : F0;
    const TopKey* top = in_b ? F.top_b : F.top_a;
    // k slots <= 2^26 (checked when the frontier is created)
    const unsigned slots = (unsigned)F.slots, total = (unsigned)k * slots;
    const unsigned long long nV = min(*F.nV, (unsigned long long)F.capacity);
    const unsigned kk = (unsigned)min((unsigned long long)k, nV);
    for (unsigned o0 = blockIdx.x * kNbThreads; o0 < total; o0 += gridDim.x * kNbThreads) {
        const unsigned r0 = o0 / slots, r1 = min(o0 + kNbThreads - 1, total - 1) / slots;
        __syncthreads();
        if (threadIdx.x <= r1 - r0 && r0 + threadIdx.x < kk)
            par_len[threadIdx.x] = decode_code(top[r0 + threadIdx.x].code, F.n_modes, par[threadIdx.x]);
        __syncthreads();
        const unsigned o = o0 + threadIdx.x;
        if (o >= total) continue;
        const unsigned r = o / slots;
        unsigned long long code = kEmpty;
        if (r < kk) {
            uint16_t nb[COMET_MAX_SEGMENTS];
            const int Ln = neighbour_r(F, par[r - r0], par_len[r - r0], (int)(o - r * slots), nb);
            if (Ln > 0) {
                comet_mode_seq q;
                q.len = (uint8_t)Ln;
                for (int i = 0; i < Ln; ++i) q.modes[i] = nb[i];
                code = encode_seq(q, F.n_modes);
                if (set_contains(F.set, F.set_mask, code))
                    code = kEmpty;  // already in V
                else
                    F.flag[o] = cand_insert(F.cand_keys, F.cand_ord, F.cand_mask, code, o);
            }
        }
        F.cand_code[o] = code;
    }
}

// Winners (the first proposal of each unseen code) keep their code, the
// other slots lose it; the winners of each block of kScan slots are counted.
__global__ void __launch_bounds__(kScan) winner_kernel(FrontierDev F0, const FrontierDev* Fs, int k) {
    launch_next();
    await_previous();
    const FrontierDev F = Fs ? Fs[blockIdx.y] : F0;
    const int64_t total = (int64_t)k * F.slots, o = blockIdx.x * (int64_t)kScan + threadIdx.x;
    if (blockIdx.x * (int64_t)kScan >= total) return;
    bool win = false;
    if (o < total && F.cand_code[o] != kEmpty) {
        const int at = F.flag[o];
        win = at >= 0 && F.cand_ord[at] == ~(unsigned int)o;
        if (!win) F.cand_code[o] = kEmpty;
    }
    const int n = __syncthreads_count(win);
    if (threadIdx.x == 0) F.counts[blockIdx.x] = n;
}

// The first `batch` winners in ordinal order (capped by the remaining
// evaluation budget) become F_{s+1}: every block adds up the counts before
// it, so the slots are placed in one parallel pass (a single-CTA scan took
// 0.7 ms over the 560,000 slots of a two-edit round).  Winners clear their
// entry of the candidate table.
__global__ void __launch_bounds__(kScan) compact_kernel(FrontierDev F0, const FrontierDev* Fs, int k, int batch_in,
                                                        int64_t budget) {
    launch_next();
    await_previous();
    __shared__ int warp_sums[32];
    const FrontierDev F = Fs ? Fs[blockIdx.y] : F0;
    const int64_t total = (int64_t)k * F.slots;
    const int blocks = (int)((total + kScan - 1) / kScan);
    if ((int)blockIdx.x >= blocks) return;
    const unsigned long long nV = min(*F.nV, (unsigned long long)F.capacity);
    int64_t cap = Fs ? F.batch : batch_in;
    if (budget > 0) cap = min(cap, budget - (int64_t)nV);
    if (cap < 0) cap = 0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // winners in the blocks before this one; block 0 adds up all of them
    int before = 0;
    const int upto = blockIdx.x == 0 ? blocks : (int)blockIdx.x;
    for (int b = threadIdx.x; b < upto; b += kScan) before += F.counts[b];
    for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
    if (lane == 0) warp_sums[w] = before;
    __syncthreads();
    before = 0;
    for (int i = 0; i < kScan / 32; ++i) before += warp_sums[i];
    __syncthreads();
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) *F.n_next = min((int64_t)before, cap);
        before = 0;
    }
    const int64_t o = blockIdx.x * (int64_t)kScan + threadIdx.x;
    const unsigned long long code = o < total ? F.cand_code[o] : kEmpty;
    const unsigned bal = __ballot_sync(0xffffffffu, code != kEmpty);
    if (lane == 0) warp_sums[w] = __popc(bal);
    __syncthreads();
    if (code == kEmpty) return;
    for (int i = 0; i < w; ++i) before += warp_sums[i];
    const int place = before + __popc(bal & ((1u << lane) - 1u));
    const int at = F.flag[o];
    F.cand_keys[at] = kEmpty;
    F.cand_ord[at] = 0u;
    if (place < cap) {
        comet_mode_seq q;
        uint16_t m[COMET_MAX_SEGMENTS];
        const int L = decode_code(code, F.n_modes, m);
        q.instance = F.instance;
        q.len = (uint8_t)L;
        for (int i = 0; i < COMET_MAX_SEGMENTS; ++i) q.modes[i] = (i < L) ? m[i] : 0;
        q.pad[0] = q.pad[1] = q.pad[2] = 0;
        F.next[place] = q;
    }
}

}  // namespace

// V's codes back into the (cleared) hash set after a checkpoint restored
// codes[0..n) and merit[0..n)
__global__ void restore_kernel(FrontierDev F, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        set_insert(F.set, F.set_mask, F.codes[i]);
}

cudaError_t launch_frontier_restore(const FrontierDev& F, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 4096);
    restore_kernel<<<blocks, threads, 0, s>>>(F, n);
    return cudaGetLastError();
}

cudaError_t launch_frontier_add(const FrontierDev& F, const comet_mode_seq* seqs, int64_t n, const int64_t* d_n,
                                const float* cost, const float* viol, float eps_feas, float merit_mu, cudaStream_t s) {
    const int64_t work = d_n ? F.batch_cap : n;
    if (work <= 0) return cudaSuccess;
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((work + threads - 1) / threads, 4096);
    add_kernel<<<blocks, threads, 0, s>>>(F, seqs, n, d_n, cost, viol, eps_feas, merit_mu);
    return cudaGetLastError();
}

// the orders of several frontiers in one launch (see add_many_kernel);
// n_max: the largest count of one frontier
cudaError_t launch_frontier_add_many(const FrontierDev* d_fs, int n_f, const comet_mode_seq* seqs, const int64_t* d_off,
                                     bool seeds, int64_t n_max, const float* cost, const float* viol, float eps_feas,
                                     float merit_mu, cudaStream_t s) {
    for (int y = 0; y < n_f; y += kMaxGridY) {
        const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>((n_max + 255) / 256, 1024)),
                        (unsigned)std::min(n_f - y, kMaxGridY));
        add_many_kernel<<<grid, 256, 0, s>>>(d_fs + y, seqs, d_off + y, seeds ? 1 : 0, cost, viol, eps_feas, merit_mu);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace {

// Top-k of one frontier (F) or of n_f frontiers (d_fs, capacities up to
// `capacity`); *in_b tells whether the keys are in top_b (else top_a).
cudaError_t topk(const FrontierDev& F, const FrontierDev* d_fs, int n_f, int64_t capacity, int k, bool* in_b,
                 cudaStream_t s) {
    int64_t runs = (capacity + kRun - 1) / kRun;
    int len = std::min(k, kRun);
    *in_b = false;
    cudaError_t e = launch_chained(topk_rank_kernel, dim3((unsigned)runs, (unsigned)n_f), kRun, 0, s, F, d_fs, k);
    for (int pass = 1; runs > 1 && e == cudaSuccess; ++pass) {
        const dim3 grid((unsigned)((runs * len + 255) / 256), (unsigned)n_f);
        e = launch_chained(topk_merge_kernel, grid, 256, 0, s, F, d_fs, pass, k);
        *in_b = pass & 1;
        runs = (runs + kMerge - 1) / kMerge;
        len = std::min(k, kMerge * len);
    }
    return e;
}

// One expansion round of one frontier (F; batch) or of n_f frontiers (d_fs,
// each with its own batch), total: the largest number of slots.
cudaError_t expand(const FrontierDev& F, const FrontierDev* d_fs, int n_f, int64_t capacity, int64_t total, int k,
                   int batch, int64_t budget, cudaStream_t s) {
    bool in_b = false;
    cudaError_t e = topk(F, d_fs, n_f, capacity, k, &in_b, s);
    if (e != cudaSuccess) return e;
    const dim3 g1((unsigned)std::min<int64_t>((total + kNbThreads - 1) / kNbThreads, 65535), (unsigned)n_f);
    const dim3 g2((unsigned)((total + kScan - 1) / kScan), (unsigned)n_f);
    if ((e = launch_chained(neighbour_kernel, g1, kNbThreads, 0, s, F, d_fs, in_b ? 1 : 0, k)) != cudaSuccess) return e;
    if ((e = launch_chained(winner_kernel, g2, kScan, 0, s, F, d_fs, k)) != cudaSuccess) return e;
    return launch_chained(compact_kernel, g2, kScan, 0, s, F, d_fs, k, batch, budget);
}

}  // namespace

const TopKey* launch_topk(const FrontierDev& F, int k, cudaStream_t s, cudaError_t* err) {
    bool in_b = false;
    *err = topk(F, nullptr, 1, F.capacity, k, &in_b, s);
    return *err != cudaSuccess ? nullptr : in_b ? F.top_b : F.top_a;
}

cudaError_t launch_topk_many(const FrontierDev* d_fs, int n_f, int64_t capacity, int k, bool* in_b, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    for (int y = 0; y < n_f && e == cudaSuccess; y += kMaxGridY)
        e = topk(FrontierDev{}, d_fs + y, std::min(n_f - y, kMaxGridY), capacity, k, in_b, s);
    return e;
}

cudaError_t launch_expand(const FrontierDev& F, int k, int batch, int64_t budget, cudaStream_t s) {
    return expand(F, nullptr, 1, F.capacity, (int64_t)k * F.slots, k, batch, budget, s);
}

cudaError_t launch_expand_many(const FrontierDev* d_fs, int n_f, int64_t capacity, int64_t slots, int k,
                               int64_t budget, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    for (int y = 0; y < n_f && e == cudaSuccess; y += kMaxGridY)
        e = expand(FrontierDev{}, d_fs + y, std::min(n_f - y, kMaxGridY), capacity, (int64_t)k * slots, k, 0, budget, s);
    return e;
}

}  // namespace comet
