// BF16 GEMM on the 5th-generation tensor cores for the learned proposal.
//
//   D[M][N] = A[M][K] . B[N][K]^T   (bf16 operands, FP32 accumulation)
//
// One CTA computes a 128 x BN tile (BN <= 64) over its share of K:
//   * warp 0, one lane: TMA producer.  Tiles of 64 K-elements (128 bytes
//     per row, the 128-byte swizzle span) of A and B are copied into a
//     4-stage shared-memory ring; each stage's full barrier counts the bytes.
//   * warp 1, one lane: MMA issuer.  Four tcgen05.mma (kind::f16, K = 16)
//     per stage accumulate into TMEM (128 lanes x BN FP32 columns); a
//     tcgen05.commit frees the stage and, after the last, signals the
//     accumulator barrier.
//   * warp 2 allocates and frees the TMEM columns.
//   * all four warps: epilogue.  Warp w reads TMEM lanes 32w..32w+31 (rows
//     of the tile) 32 columns at a time with tcgen05.ld and applies the fused
//     epilogue (bias, GELU, GELU' gating, the loss, BF16 conversion, the
//     transposed copy the weight-gradient GEMM consumes, or split-K atomics):
//     aligned rows from registers, a row per lane; ragged blocks and split-K
//     sums turned around in shared memory, lanes along a row.
//
// The kernels are chained (launch.h): the successor may start once the TMEM
// columns are held, and nothing global is touched before await_previous().
//
// Every mbarrier wait is bounded (about one second of clock cycles); when
// one runs out the CTA records the failure in the error flag, skips the rest
// of its work, waits (bounded) for the copies it issued and frees its TMEM.
#include "launch.h"
#include "mlp_internal.h"

#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <string.h>

#include <algorithm>
#include <mutex>

namespace comet {
namespace mlp {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;           // bf16 elements per 128-byte swizzle row
constexpr int kStages = 4;
constexpr int kThreads = 128;
constexpr int kMaxBN = 64;  // column tile: more CTAs for the small GEMMs of the MLP
constexpr long long kWaitCycles = 2000000000ll;  // ~1 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity; false if it ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile stored as rows
// of 128 bytes with the 128-byte swizzle (the layout TMA writes with
// CU_TENSOR_MAP_SWIZZLE_128B): 8-row groups 1024 bytes apart (stride byte
// offset), leading byte offset unused, descriptor version 1, swizzle mode 2.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint16_t to_bf16(float x) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// GELU in the tanh form of Hendrycks and Gimpel,
//   0.5 x (1 + tanh(a (x + b x^3))), a = sqrt(2 / pi), b = 0.044715,
// with the hardware tanh approximation (relative error about 2^-11, below
// the BF16 rounding of the stored activations)
__device__ __forceinline__ float tanh_hw(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr float kGeluA = 0.79788456080286536f;  // sqrt(2 / pi)
constexpr float kGeluB = 0.044715f;

__device__ __forceinline__ float gelu_f(float x) {
    const float t = tanh_hw(kGeluA * (x + kGeluB * x * x * x));
    return 0.5f * x * (1.f + t);
}

__device__ __forceinline__ float gelu_grad_f(float x) {
    const float t = tanh_hw(kGeluA * (x + kGeluB * x * x * x));
    return 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * kGeluA * (1.f + 3.f * kGeluB * x * x);
}

struct __align__(8) Barriers {
    uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t accum;
    uint32_t tmem_base;
    uint32_t failed;
};

// What a tile's epilogue may take from the operands' alignment: 16-byte
// accesses along a row (decided on the host).
struct Tile {
    int M, N, m0, n0, k_begin, k_len, bn, tmem_cols, vec;
};

// Epilogue of one 32 x 32 block in the accumulator's own layout: a lane holds
// 32 consecutive columns of its row, so that rows move as 16-byte accesses
// and the transposed copy as 64-byte runs over the lanes (rows), with nothing
// turned around in shared memory and all operand loads issued before the
// first use.  A training step of 4,096 rows, per launch: 14.7 -> 9.0 us (GELU
// with its three outputs), 42 -> 9.5 us (GELU' gating, whose loads were one
// dependent access per row).
template <int KIND>
__device__ __forceinline__ void epilogue_rows(const Epilogue& ep, uint32_t taddr, int row, int nb, int ncol,
                                              bool row_ok, float& loss) {
    float v[32], x[32];
    // 4 q < ncol only bites for kEpiLoss (N a multiple of 16); the other kinds
    // come here with whole blocks
    const bool whole = KIND != kEpiLoss;
    if (KIND == kEpiGeluGrad) {
        const float4* z = reinterpret_cast<const float4*>(ep.z_in + (int64_t)row * ep.ld_z + nb);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 t = row_ok ? z[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            x[4 * q] = t.x, x[4 * q + 1] = t.y, x[4 * q + 2] = t.z, x[4 * q + 3] = t.w;
        }
    } else if (ep.bias) {
        const float4* z = reinterpret_cast<const float4*>(ep.bias + nb);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 t = whole || 4 * q < ncol ? z[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            x[4 * q] = t.x, x[4 * q + 1] = t.y, x[4 * q + 2] = t.z, x[4 * q + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = 0.f;
    }
    float t[KIND == kEpiLoss ? 32 : 1], om[KIND == kEpiLoss ? 32 : 1];
    if constexpr (KIND == kEpiLoss) {
        const float4* tp = reinterpret_cast<const float4*>(ep.target + (int64_t)row * ep.ld_z + nb);
        const float4* op = reinterpret_cast<const float4*>(ep.weight + (int64_t)row * ep.ld_z + nb);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const bool ok = row_ok && 4 * q < ncol;
            const float4 a = ok ? tp[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 b = ok ? op[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            t[4 * q] = a.x, t[4 * q + 1] = a.y, t[4 * q + 2] = a.z, t[4 * q + 3] = a.w;
            om[4 * q] = b.x, om[4 * q + 1] = b.y, om[4 * q + 2] = b.z, om[4 * q + 3] = b.w;
        }
    }
    tmem_ld32(taddr, v);
    if (!row_ok) return;
    uint32_t hb[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        if constexpr (KIND == kEpiStore) {
            v[j] += x[j];
        } else if constexpr (KIND == kEpiBiasGelu) {
            v[j] += x[j];
            hb[j] = to_bf16(gelu_f(v[j]));
        } else if constexpr (KIND == kEpiGeluGrad) {
            hb[j] = to_bf16(v[j] * gelu_grad_f(x[j]));
        } else if constexpr (KIND == kEpiLoss) {
            // dL/dY = (2/B) Omega (Y - T), and the row's share of the loss
            const float d = v[j] + x[j] - t[j], w = om[j];
            if (j < ncol) loss += w * d * d;
            hb[j] = to_bf16(2.f * w * d * ep.inv_b);
        }
    }
    if (KIND == kEpiStore || (KIND == kEpiBiasGelu && ep.out_f32)) {
        float4* o = reinterpret_cast<float4*>(ep.out_f32 + (int64_t)row * ep.ld_out + nb);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    if constexpr (KIND != kEpiStore && KIND != kEpiAtomicAdd) {
        if (ep.h) {
            uint4* o = reinterpret_cast<uint4*>(ep.h + (int64_t)row * ep.ld_h + nb);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = hb[8 * q + 2 * i] | (hb[8 * q + 2 * i + 1] << 16);
                if (whole || 8 * q < ncol) o[q] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        if (ep.h_t) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (whole || j < ncol) ep.h_t[(int64_t)(nb + j) * ep.ld_ht + row] = (uint16_t)hb[j];
        }
    }
}

// One CTA's tile of D = A B^T: the pipeline and the epilogue.
template <int KIND>
__device__ __forceinline__ void gemm_tile(const CUtensorMap* map_a, const CUtensorMap* map_b, const Tile& T,
                                          const Epilogue& ep) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    const int M = T.M, N = T.N, m0 = T.m0, n0 = T.n0, bn = T.bn;
    const uint32_t a_bytes = BM * BK * 2;
    const uint32_t b_bytes = (uint32_t)bn * BK * 2;
    const uint32_t stage_bytes = a_bytes + b_bytes;
    Barriers* bars = reinterpret_cast<Barriers*>(smem + kStages * stage_bytes);
    const uint32_t s_base = smem_u32(smem);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = (T.k_len + BK - 1) / BK;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&bars->full[s]), 1);
            mbar_init(smem_u32(&bars->empty[s]), 1);
        }
        mbar_init(smem_u32(&bars->accum), 1);
        bars->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&bars->tmem_base)),
                     "r"(T.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    launch_next();
    await_previous();

    if (warp == 0 && lane == 0) {
        // ---- producer
        int issued = 0;
        for (int i = 0; i < nkb; ++i) {
            const int s = i % kStages;
            const uint32_t ph = (uint32_t)(i / kStages) & 1u;
            if (i >= kStages && !mbar_wait(smem_u32(&bars->empty[s]), ph ^ 1u)) {
                atomicExch(&bars->failed, 1u);
                break;
            }
            if (*(volatile uint32_t*)&bars->failed) break;
            const uint32_t full = smem_u32(&bars->full[s]);
            mbar_expect_tx(full, stage_bytes);
            const int kx = T.k_begin + i * BK;
            tma_load_2d(s_base + s * stage_bytes, map_a, kx, m0, full);
            tma_load_2d(s_base + s * stage_bytes + a_bytes, map_b, kx, n0, full);
            ++issued;
        }
        if (*(volatile uint32_t*)&bars->failed) {
            // wait (bounded) for the copies still in flight before the CTA
            // can release its shared memory
            for (int i = (issued > kStages ? issued - kStages : 0); i < issued; ++i)
                mbar_wait(smem_u32(&bars->full[i % kStages]), (uint32_t)(i / kStages) & 1u);
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        const uint32_t idesc = instr_desc(BM, bn);
        bool ok = true;
        for (int i = 0; i < nkb && ok; ++i) {
            const int s = i % kStages;
            const uint32_t ph = (uint32_t)(i / kStages) & 1u;
            if (!mbar_wait(smem_u32(&bars->full[s]), ph)) {
                atomicExch(&bars->failed, 1u);
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t a = s_base + s * stage_bytes, b = a + a_bytes;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
                mma_bf16(tmem, smem_desc(a + kk * 32), smem_desc(b + kk * 32), idesc, (i > 0 || kk > 0) ? 1u : 0u);
            mma_commit(smem_u32(&bars->empty[s]));
        }
        mma_commit(smem_u32(&bars->accum));
    }
    __syncwarp();

    // ---- epilogue: all warps
    const bool have = mbar_wait(smem_u32(&bars->accum), 0);
    if (!have) atomicExch(&bars->failed, 1u);
    tc_fence_after();
    __syncwarp();
    const bool run = __all_sync(0xffffffffu, have && !*(volatile uint32_t*)&bars->failed);
    float loss = 0.f;
    if (run) {
        float* st1 = reinterpret_cast<float*>(smem) + warp * (2 * 32 * 33);
        float* st2 = st1 + 32 * 33;
        const int row0 = m0 + warp * 32;
        for (int c0 = 0; c0 < bn; c0 += 32) {
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
            const int nb = n0 + c0;
            if (nb >= N) break;
            if (KIND == kEpiLoss || (KIND != kEpiAtomicAdd && T.vec && nb + 32 <= N)) {
                const int row = row0 + lane;
                epilogue_rows<KIND>(ep, taddr, row, nb, min(32, N - nb), row < M, loss);
                continue;
            }
            // A block of ragged columns or unaligned rows, and the split-K
            // sums: turned around in shared memory (the pipeline stages are
            // free once the accumulator is complete), so that row-major
            // outputs are written with lanes along a row and the transposed
            // copy with lanes along a column.  Warp w stages in its own two
            // 32 x 33 tiles (raw accumulator, result).
            float v[32];
            tmem_ld32(taddr, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) st1[lane * 33 + j] = v[j];
            __syncwarp();
            // lanes along a row: column nb + lane
            const int col = nb + lane;
            const bool col_ok = col < N;
            const float bias = (KIND != kEpiAtomicAdd && ep.bias && col_ok) ? ep.bias[col] : 0.f;
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
                const int row = row0 + r;
                const bool ok = col_ok && row < M;
                const float a = st1[r * 33 + lane];
                float res = 0.f;
                if (KIND == kEpiStore) {
                    if (ok) ep.out_f32[(int64_t)row * ep.ld_out + col] = a + bias;
                } else if (KIND == kEpiAtomicAdd) {
                    // the last column of a weight gradient with a row of ones
                    // under its second operand is the split's bias gradient,
                    // the only sum that its zeroed place gets (a branch to a
                    // plain store costs the launch 1.5 us)
                    if (ok)
                        atomicAdd(ep.bias_grad && col == N - 1 ? ep.bias_grad + row
                                                               : ep.out_f32 + (int64_t)row * ep.ld_out + col,
                                  a);
                } else if (KIND == kEpiBiasGelu) {
                    const float z = a + bias;
                    if (ok && ep.out_f32) ep.out_f32[(int64_t)row * ep.ld_out + col] = z;
                    res = gelu_f(z);
                } else {  // kEpiGeluGrad
                    const float z = ok ? ep.z_in[(int64_t)row * ep.ld_z + col] : 0.f;
                    res = a * gelu_grad_f(z);
                }
                if (KIND == kEpiBiasGelu || KIND == kEpiGeluGrad) {
                    const uint16_t hb = to_bf16(res);
                    if (ok && ep.h) ep.h[(int64_t)row * ep.ld_h + col] = hb;
                    st2[r * 33 + lane] = __uint_as_float((uint32_t)hb);
                }
            }
            __syncwarp();
            if ((KIND == kEpiBiasGelu || KIND == kEpiGeluGrad) && ep.h_t) {
                // lanes along a column of the transposed copy: row row0 + lane
                const int row = row0 + lane;
                if (row < M) {
                    const int nv = min(32, N - nb);
                    for (int j = 0; j < nv; ++j)
                        ep.h_t[(int64_t)(nb + j) * ep.ld_ht + row] = (uint16_t)__float_as_uint(st2[lane * 33 + j]);
                }
            }
            __syncwarp();
        }
    }
    if (KIND == kEpiLoss) {
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (lane == 0) atomicAdd(ep.loss, loss * ep.inv_b);
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *ep.step += 1;
    }
    if (*(volatile uint32_t*)&bars->failed && threadIdx.x == 0 && ep.err) atomicExch(ep.err, 1);
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T.tmem_cols) : "memory");
    }
}

template <int KIND>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_bf16_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M,
                     int N, int K, int k_chunk, int bn, int tmem_cols, int vec, Epilogue ep) {
    const int k_begin = blockIdx.z * k_chunk;
    gemm_tile<KIND>(&map_a, &map_b,
                    Tile{M, N, (int)blockIdx.x * BM, (int)blockIdx.y * bn, k_begin, min(k_chunk, K - k_begin), bn,
                         tmem_cols, vec},
                    ep);
}

// The weight and bias gradients of all layers in one launch: blockIdx.x runs
// over the (layer, row tile, column tile) triples, blockIdx.y over the splits
// of the batch.
struct DwMaps {
    CUtensorMap a[kDwMax], b[kDwMax];
};
struct DwParams {
    int n, K, k_chunk, first[kDwMax + 1], M[kDwMax], N[kDwMax], cols[kDwMax];
    float* dw[kDwMax];
    float* db[kDwMax];
    int64_t ld_db;
    int* err;
};

__global__ void __launch_bounds__(kThreads, 1) dw_kernel(const __grid_constant__ DwMaps maps, const DwParams P) {
    int l = 0;
    while (l + 1 < P.n && (int)blockIdx.x >= P.first[l + 1]) ++l;
    const int t = (int)blockIdx.x - P.first[l];
    const int k_begin = blockIdx.y * P.k_chunk;
    Epilogue ep;
    ep.kind = kEpiAtomicAdd;
    ep.out_f32 = P.dw[l];
    ep.ld_out = P.N[l] - 1;
    ep.bias_grad = P.db[l] + blockIdx.y * P.ld_db;
    ep.err = P.err;
    gemm_tile<kEpiAtomicAdd>(&maps.a[l], &maps.b[l],
                             Tile{P.M[l], P.N[l], t / P.cols[l] * BM, t % P.cols[l] * kMaxBN, k_begin,
                                  min(P.k_chunk, P.K - k_begin), kMaxBN, kMaxBN, 0},
                             ep);
}

// ------------------------------------------------------------------------
// Fused forward pass of the 4-layer MLP (in_dim <= 256, width 256, any
// out_dim): persistent CTAs walk units of a 128-row tile and a share of the
// output's 256-column blocks; the layers are chained through two 256-column
// TMEM accumulators and a 64 KB activation tile in shared memory, so a tile
// never leaves the SM between layers.  Warps 0..15: epilogue (warp w reads
// TMEM lanes 32 (w mod 4)..); warp 16, one lane: TMA producer (the X tile,
// and the weights as 64-column K slices of 256 rows through a ring); warp 17,
// one lane: MMA issuer.
//
// A hidden layer's epilogue writes bias + GELU as BF16 into the activation
// tile in the 128-byte-swizzled K-major layout the next tcgen05.mma reads
// (16-byte chunk c of row r at chunk c ^ (r mod 8)), one 64-column K slice
// after the other over all 16 warps (16 columns each); the next layer's MMAs
// start on a slice as soon as it is ready, into the other accumulator, so
// that a layer costs its epilogue and one slice's MMA instead of the sum of
// both.  An output block's MMAs run under the previous block's stores.  What
// bounds a tile is the epilogue's FP32 arithmetic (GELU on pairs of values by
// f32x2 instructions, results unchanged).  20,736 rows 64 -> 256: 40 us with
// one accumulator, scalar GELU and layers in sequence, 29 us now.  The box
// flip's 192 -> 1,088 (8,192 rows) took 51 us as four GEMM launches, 24 us
// now; with fewer tiles than SMs the output blocks are split over CTAs, each
// repeating the hidden layers (cheaper than idle SMs).

constexpr int kFEpiWarps = 16;
constexpr int kFThreads = (kFEpiWarps + 2) * 32;
constexpr int kFRing = 3;                    // weight slices in flight (2 when in_dim > 192)
constexpr uint32_t kWStage = 256 * BK * 2;   // 32 KB: one K slice of a weight
constexpr uint32_t kXBlock = BM * BK * 2;    // 16 KB: one K slice of a tile

struct __align__(8) FusedBars {
    uint64_t x_full, x_free, drain;
    uint64_t acc_full[2], acc_free[2], h_ready[4];
    uint64_t w_full[kFRing], w_empty[kFRing];
    uint32_t tmem_base, failed;
};

struct FusedParams {
    const float* bias[4];
    float* y;
    int64_t ld_y;
    int M, in_dim, out_dim, ring, nsplit;
    int* err;
};

// Bounded wait that also ends when another role of the CTA has given up.
__device__ __forceinline__ bool fused_wait(uint32_t bar, uint32_t parity, volatile uint32_t* failed) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*failed) return false;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}

// 16 consecutive FP32 columns of this thread's TMEM lane (no wait)
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t r[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// two FP32 values in one register pair
__device__ __forceinline__ uint64_t f2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_get(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// BF16 pair of gelu_f(v + bias) for two values, the same operations as
// gelu_f in the same order
__device__ __forceinline__ uint32_t gelu_pair(uint64_t v, uint64_t bias) {
    const uint64_t x = f2_add(v, bias);
    const uint64_t u = f2_mul(f2_mul(f2(kGeluB, kGeluB), x), x);
    float a, b;
    f2_get(f2_mul(f2(kGeluA, kGeluA), f2_fma(u, x, x)), a, b);
    const uint64_t t = f2_add(f2(1.f, 1.f), f2(tanh_hw(a), tanh_hw(b)));
    f2_get(f2_mul(f2_mul(f2(0.5f, 0.5f), x), t), a, b);
    uint32_t pk;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk) : "f"(b), "f"(a));
    return pk;
}

__global__ void __launch_bounds__(kFThreads, 1)
    mlp_fused_forward_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w0,
                             const __grid_constant__ CUtensorMap map_w1, const __grid_constant__ CUtensorMap map_w2,
                             const __grid_constant__ CUtensorMap map_w3, const FusedParams fp) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    const int n_xkb = fp.in_dim / BK;                             // 1..4 K slices of X
    const int ring = fp.ring;
    uint8_t* xs = smem;                                           // n_xkb x 16 KB
    uint8_t* hs = xs + n_xkb * kXBlock;                           // 4 x 16 KB activations
    uint8_t* ws = hs + 4 * kXBlock;                               // ring x 32 KB weights
    float* bs = reinterpret_cast<float*>(ws + ring * kWStage);    // 3 x 256 biases
    FusedBars* bars = reinterpret_cast<FusedBars*>(bs + 3 * 256);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_ob = (fp.out_dim + 255) / 256;                    // output blocks
    const int n_units = (fp.M + BM - 1) / BM * fp.nsplit;
    const CUtensorMap* wmap[4] = {&map_w0, &map_w1, &map_w2, &map_w3};

    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars->x_full), 1);
        mbar_init(smem_u32(&bars->x_free), 1);
        mbar_init(smem_u32(&bars->drain), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars->acc_full[i]), 1);
            mbar_init(smem_u32(&bars->acc_free[i]), kFEpiWarps);
        }
        for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&bars->h_ready[i]), kFEpiWarps);
        for (int s = 0; s < ring; ++s) {
            mbar_init(smem_u32(&bars->w_full[s]), 1);
            mbar_init(smem_u32(&bars->w_empty[s]), 1);
        }
        bars->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&bars->tmem_base)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    volatile uint32_t* failed = &bars->failed;
    launch_next();
    await_previous();
    for (int t = threadIdx.x; t < 3 * 256; t += kFThreads) bs[t] = fp.bias[t >> 8][t & 255];
    __syncthreads();

    // A unit's steps: the hidden layers 0..2, then its output blocks split,
    // split + nsplit, ...; step number g (over all units) uses accumulator
    // g & 1, whose barriers complete once per use
    if (warp == kFEpiWarps) {
        if (lane == 0) {
            // ---- producer
            uint32_t n_w = 0;  // weight slices issued
            int it = 0;
            bool ok = true;
            auto slice = [&](int l, int kb, int row) {
                const int s = (int)(n_w % ring);
                const uint32_t use = n_w / ring;
                if (n_w >= (uint32_t)ring && !fused_wait(smem_u32(&bars->w_empty[s]), (use & 1u) ^ 1u, failed))
                    return false;
                const uint32_t fb = smem_u32(&bars->w_full[s]);
                mbar_expect_tx(fb, kWStage);
                tma_load_2d(smem_u32(ws) + s * kWStage, wmap[l], kb * BK, row, fb);
                ++n_w;
                return true;
            };
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x, ++it) {
                const int tile = u / fp.nsplit, split = u % fp.nsplit;
                ok = it == 0 || fused_wait(smem_u32(&bars->x_free), (uint32_t)(it - 1) & 1u, failed);
                if (!ok) break;
                const uint32_t xb = smem_u32(&bars->x_full);
                mbar_expect_tx(xb, (uint32_t)n_xkb * kXBlock);
                for (int kb = 0; kb < n_xkb; ++kb)
                    tma_load_2d(smem_u32(xs) + kb * kXBlock, &map_x, kb * BK, tile * BM, xb);
                for (int l = 0; l < 3 && ok; ++l)
                    for (int kb = 0; kb < (l == 0 ? n_xkb : 4) && ok; ++kb) ok = slice(l, kb, 0);
                for (int b = split; b < n_ob && ok; b += fp.nsplit)
                    for (int kb = 0; kb < 4 && ok; ++kb) ok = slice(3, kb, 256 * b);
            }
            if (!ok) {
                // wait (bounded) for the copies in flight before the CTA can
                // release its shared memory
                *failed = 1u;
                for (uint32_t i = n_w > (uint32_t)ring ? n_w - ring : 0; i < n_w; ++i)
                    mbar_wait(smem_u32(&bars->w_full[i % ring]), (i / ring) & 1u);
                if (it > 0) mbar_wait(smem_u32(&bars->x_full), (uint32_t)(it - 1) & 1u);
            }
        }
    } else if (warp == kFEpiWarps + 1) {
        if (lane == 0) {
            // ---- MMA issuer
            uint32_t n_w = 0, g = 0, hc = 0;  // weight slices used, steps, hidden layers
            int it = 0;
            bool ok = true;
            // step of n_kb K slices with A at `a`; h_wait: the slices of A are
            // the hidden layer before (number hc - 1), taken as they get ready
            auto step = [&](uint32_t a, int n_kb, int n_cols, bool h_wait) {
                const uint32_t acc = g & 1u, idesc = instr_desc(BM, n_cols);
                if (g >= 2 && !fused_wait(smem_u32(&bars->acc_free[acc]), ((g >> 1) - 1u) & 1u, failed)) return false;
                for (int kb = 0; kb < n_kb; ++kb, ++n_w) {
                    const int s = (int)(n_w % ring);
                    if (h_wait && !fused_wait(smem_u32(&bars->h_ready[kb]), (hc - 1u) & 1u, failed)) return false;
                    if (!fused_wait(smem_u32(&bars->w_full[s]), (n_w / ring) & 1u, failed)) return false;
                    tc_fence_after();
                    const uint32_t ak = a + kb * kXBlock, b = smem_u32(ws) + s * kWStage;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_bf16(tmem + acc * 256, smem_desc(ak + kk * 32), smem_desc(b + kk * 32), idesc,
                                 (kb > 0 || kk > 0) ? 1u : 0u);
                    mma_commit(smem_u32(&bars->w_empty[s]));
                }
                mma_commit(smem_u32(&bars->acc_full[acc]));
                ++g;
                return true;
            };
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x, ++it) {
                const int split = u % fp.nsplit;
                ok = fused_wait(smem_u32(&bars->x_full), (uint32_t)it & 1u, failed);
                if (ok) ok = step(smem_u32(xs), n_xkb, 256, false);
                if (!ok) break;
                mma_commit(smem_u32(&bars->x_free));
                ++hc;
                for (int l = 1; l < 3 && ok; ++l, ++hc) ok = step(smem_u32(hs), 4, 256, true);
                for (int b = split; b < n_ob && ok; b += fp.nsplit)
                    ok = step(smem_u32(hs), 4, min(256, fp.out_dim - 256 * b), b == split);
            }
            if (!ok) {
                // the tensor cores are done with shared memory and TMEM
                // (bounded) before the CTA releases them
                *failed = 1u;
                mma_commit(smem_u32(&bars->drain));
                mbar_wait(smem_u32(&bars->drain), 0);
            }
        }
    } else {
        // ---- epilogue warps: row r = 32 (warp mod 4) + lane of the tile
        const int quarter = warp & 3, part = warp >> 2;
        const int r = quarter * 32 + lane;
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        uint32_t g = 0;
        bool ok = true;
        auto wait_acc = [&]() {
            const bool have = fused_wait(smem_u32(&bars->acc_full[g & 1u]), (g >> 1) & 1u, failed);
            tc_fence_after();
            return (bool)__all_sync(0xffffffffu, have);
        };
        // the accumulator's values are in registers
        auto free_acc = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars->acc_free[g & 1u]));
        };
        for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
            const int tile = u / fp.nsplit, split = u % fp.nsplit;
            for (int l = 0; l < 3 && ok; ++l) {
                ok = wait_acc();
                if (!ok) break;
                uint32_t v[4][16];
                const uint32_t acc = tmem + lanes + (g & 1u) * 256 + 16 * part;
#pragma unroll
                for (int s = 0; s < 4; ++s) tmem_ld16_nowait(acc + 64 * s, v[s]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                free_acc();
                const float* bias = bs + 256 * l + 16 * part;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    // 16 BF16 = two 16-byte chunks of row r of K slice s,
                    // placed by the 128-byte swizzle
                    uint32_t pk[8];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 bv = *reinterpret_cast<const float4*>(bias + 64 * s + 4 * q);
                        pk[2 * q] = gelu_pair(f2(__uint_as_float(v[s][4 * q]), __uint_as_float(v[s][4 * q + 1])),
                                              f2(bv.x, bv.y));
                        pk[2 * q + 1] = gelu_pair(
                            f2(__uint_as_float(v[s][4 * q + 2]), __uint_as_float(v[s][4 * q + 3])), f2(bv.z, bv.w));
                    }
                    uint8_t* blk = hs + s * kXBlock + r * 128;
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        *reinterpret_cast<uint4*>(blk + ((2 * part + q) ^ (r & 7)) * 16) =
                            make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
                    // make the writes visible to the tensor cores, release the slice
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bars->h_ready[s]));
                }
                ++g;
            }
            for (int b = split; b < n_ob && ok; b += fp.nsplit) {
                ok = wait_acc();
                if (!ok) break;
                const int ncol = min(256, fp.out_dim - 256 * b);
                const int row0 = tile * BM + quarter * 32 + (lane & ~7), j8 = lane & 7;
#pragma unroll 1
                for (int c0 = 64 * part; c0 < 64 * part + 64; c0 += 32) {
                    if (c0 >= ncol) break;
                    const bool col_ok = c0 + 4 * j8 < ncol;  // out_dim is a multiple of 16
                    const int64_t col = 256 * (int64_t)b + c0 + 4 * j8;
                    float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (col_ok) bv = *reinterpret_cast<const float4*>(fp.bias[3] + col);
                    float v[32];
                    tmem_ld32(tmem + lanes + (g & 1u) * 256 + (uint32_t)c0, v);
                    // 8 lanes turn their 8 x 8 groups of four columns around
                    // (three exchanges), so that a store writes whole 128-byte
                    // lines: lane j then holds columns 4 j .. 4 j + 3 of the
                    // 8 rows
#pragma unroll
                    for (int d = 1; d < 8; d <<= 1) {
                        const bool up = j8 & d;
#pragma unroll
                        for (int p = 0; p < 8; ++p) {
                            if (p & d) continue;
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                float &lo = v[4 * p + i], &hi = v[4 * (p | d) + i];
                                const float got = __shfl_xor_sync(0xffffffffu, up ? lo : hi, d);
                                if (up) lo = got; else hi = got;
                            }
                        }
                    }
                    if (col_ok) {
                        float* y = fp.y + (int64_t)row0 * fp.ld_y + col;
#pragma unroll
                        for (int p = 0; p < 8; ++p)
                            if (row0 + p < fp.M)
                                *reinterpret_cast<float4*>(y + (int64_t)p * fp.ld_y) =
                                    make_float4(v[4 * p] + bv.x, v[4 * p + 1] + bv.y, v[4 * p + 2] + bv.z,
                                                v[4 * p + 3] + bv.w);
                    }
                }
                free_acc();
                ++g;
            }
        }
        if (!ok) *failed = 1u;
    }
    if (*failed && threadIdx.x == 0 && fp.err) atomicExch(fp.err, 1);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

int fused_ring(int in_dim) { return in_dim > 192 ? 2 : kFRing; }

size_t fused_smem_bytes(int in_dim) {
    return 1024 + (in_dim / BK + 4) * (size_t)kXBlock + fused_ring(in_dim) * (size_t)kWStage + 3 * 256 * sizeof(float) +
           sizeof(FusedBars) + 64;
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

void resolve_encode() {
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
}

// 2-D tensor map of the leading rows x cols block of a row-major bf16
// matrix, box = 64 columns x box_rows; reads past the block return zeros
bool make_map(CUtensorMap* map, const Mat& m, int64_t rows, int64_t cols, int box_rows) {
    resolve_encode();
    if (!g_encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)m.ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(m.ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// dynamic shared memory of a launch with column tile bn (at most two CTAs
// fit on an SM, holding 2 x 64 of its 512 TMEM columns)
size_t smem_request(int bn) {
    return 1024 + (size_t)kStages * (BM * BK * 2 + (size_t)bn * BK * 2) + sizeof(Barriers) + 64;
}

int g_raised[64] = {};
std::mutex g_raise_mu;

}  // namespace

cudaError_t gemm_prepare() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const int need = (int)smem_request(kMaxBN);
    std::lock_guard<std::mutex> lk(g_raise_mu);
    if (dev < 64 && g_raised[dev] >= need) return cudaSuccess;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    e = cudaFuncSetAttribute(gemm_bf16_kernel<kEpiStore>, at, need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_kernel<kEpiBiasGelu>, at, need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_kernel<kEpiGeluGrad>, at, need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_kernel<kEpiAtomicAdd>, at, need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_kernel<kEpiLoss>, at, need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dw_kernel, at, need);
    if (e == cudaSuccess && dev < 64) g_raised[dev] = need;
    return e;
}

bool tensor_maps_available() {
    resolve_encode();
    return g_encode != nullptr;
}

// whether every row access of the epilogue is 16-byte aligned
static int rows_vectorise(const Epilogue& ep) {
    auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    const bool f = !ep.out_f32 || (al(ep.out_f32) && ep.ld_out % 4 == 0);
    const bool h = !ep.h || (al(ep.h) && ep.ld_h % 8 == 0);
    const bool z = !ep.z_in || (al(ep.z_in) && ep.ld_z % 4 == 0);
    const bool t = ep.kind != kEpiLoss || (al(ep.target) && al(ep.weight) && ep.ld_z % 4 == 0);
    return f && h && z && t && (!ep.bias || al(ep.bias));
}

cudaError_t gemm_bf16(const Mat& A, const Mat& B, int64_t M, int N, int K, int k_splits, const Epilogue& ep,
                      cudaStream_t s) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (K <= 0 || k_splits < 1 || M > (int64_t)INT32_MAX) return cudaErrorInvalidValue;
    if ((reinterpret_cast<uintptr_t>(A.ptr) & 15u) || (reinterpret_cast<uintptr_t>(B.ptr) & 15u) || (A.ld & 7) ||
        (B.ld & 7) || A.cols < K || B.cols < K || A.rows < M || B.rows < N)
        return cudaErrorInvalidValue;
    if (k_splits > 1 && ep.kind != kEpiAtomicAdd) return cudaErrorInvalidValue;
    // column tile: N rounded up to 16, at most kMaxBN; TMEM columns: a power
    // of two >= 32 covering the tile
    const int n16 = (N + 15) / 16 * 16;
    const int bn = n16 <= kMaxBN ? n16 : kMaxBN;
    int tmem_cols = 32;
    while (tmem_cols < bn) tmem_cols <<= 1;
    int k_chunk = (K + k_splits - 1) / k_splits;
    k_chunk = (k_chunk + BK - 1) / BK * BK;
    const int splits = (K + k_chunk - 1) / k_chunk;
    CUtensorMap ma, mb;
    // the maps cover exactly M x K and N x K: padding rows and columns of the
    // buffers are never read (the copies fill them with zeros)
    if (!make_map(&ma, A, M, K, BM) || !make_map(&mb, B, N, K, bn)) return cudaErrorInvalidValue;
    const size_t smem_req = smem_request(bn);
    cudaError_t e = gemm_prepare();
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)((N + bn - 1) / bn), (unsigned)splits);
    const int vec = rows_vectorise(ep);
    if (ep.kind == kEpiLoss && (!vec || N % 16)) return cudaErrorInvalidValue;
#define COMET_GEMM(kind) \
    e = launch_chained(gemm_bf16_kernel<kind>, grid, kThreads, smem_req, s, ma, mb, (int)M, N, K, k_chunk, bn, \
                       tmem_cols, vec, ep)
    switch (ep.kind) {
        case kEpiStore: COMET_GEMM(kEpiStore); break;
        case kEpiBiasGelu: COMET_GEMM(kEpiBiasGelu); break;
        case kEpiGeluGrad: COMET_GEMM(kEpiGeluGrad); break;
        case kEpiAtomicAdd: COMET_GEMM(kEpiAtomicAdd); break;
        case kEpiLoss: COMET_GEMM(kEpiLoss); break;
        default: return cudaErrorInvalidValue;
    }
#undef COMET_GEMM
    return e;
}

// tiles of a layer's gradient with its bias column: rows x columns
static int dw_cols(const DwLayer& L) { return (L.din + kMaxBN) / kMaxBN; }
static int dw_tiles(const DwLayer& L) { return (L.dout + BM - 1) / BM * dw_cols(L); }

// rows of a split: one wave of two CTAs per SM, at least 256 rows each
static int dw_chunk(const DwLayer* layers, int n, int64_t K, int num_sms) {
    int tiles = 0;
    for (int l = 0; l < n; ++l) tiles += dw_tiles(layers[l]);
    const int64_t splits = std::max<int64_t>(1, std::min<int64_t>(2 * num_sms / tiles, K / 256));
    return (int)(((K + splits - 1) / splits + BK - 1) / BK * BK);
}

int dw_splits(const DwLayer* layers, int n, int64_t K, int num_sms) {
    const int chunk = dw_chunk(layers, n, K, num_sms);
    return (int)((K + chunk - 1) / chunk);
}

// splits <= max(1, 2 num_sms / tiles) (whole chunks cover K with no more), and
// a tile has at most BM of the outputs
int64_t dw_parts_max(int64_t sum_dout, int num_sms) { return std::max<int64_t>(sum_dout, 2 * (int64_t)num_sms * BM); }

cudaError_t dw_bf16(const DwLayer* layers, int n, int64_t K, int64_t ld_db, int num_sms, int* err, cudaStream_t s) {
    if (n < 1 || n > kDwMax || K < 1 || K > (int64_t)INT32_MAX) return cudaErrorInvalidValue;
    DwMaps maps;
    DwParams P;
    memset(&P, 0, sizeof(P));
    P.n = n;
    P.K = (int)K;
    P.ld_db = ld_db;
    P.err = err;
    for (int l = 0; l < n; ++l) {
        const DwLayer& L = layers[l];
        if ((reinterpret_cast<uintptr_t>(L.g_t) & 15u) || (reinterpret_cast<uintptr_t>(L.h_t) & 15u) || (L.ld & 7) ||
            L.ld < K)
            return cudaErrorInvalidValue;
        if (!make_map(&maps.a[l], Mat{L.g_t, L.dout, K, L.ld}, L.dout, K, BM) ||
            !make_map(&maps.b[l], Mat{L.h_t, L.din + 1, K, L.ld}, L.din + 1, K, kMaxBN))
            return cudaErrorInvalidValue;
        P.M[l] = L.dout;
        P.N[l] = L.din + 1;
        P.cols[l] = dw_cols(L);
        P.dw[l] = L.dw;
        P.db[l] = L.db;
        P.first[l + 1] = P.first[l] + dw_tiles(L);
    }
    P.k_chunk = dw_chunk(layers, n, K, num_sms);
    const cudaError_t e = gemm_prepare();
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)P.first[n], (unsigned)dw_splits(layers, n, K, num_sms));
    return launch_chained(dw_kernel, grid, kThreads, smem_request(kMaxBN), s, maps, P);
}

bool fused_forward_fits(int in_dim, int width, int out_dim) {
    return width == 256 && in_dim >= 64 && in_dim <= 256 && in_dim % 64 == 0 && out_dim >= 16 && out_dim % 16 == 0;
}

cudaError_t mlp_forward_fused(const uint16_t* x, int64_t M, int in_dim, const uint16_t* const w[4], int out_dim,
                              const float* const bias[4], float* y, int64_t ld_y, int* err, int num_sms,
                              cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    if (!fused_forward_fits(in_dim, 256, out_dim) || M > (int64_t)INT32_MAX - BM) return cudaErrorInvalidValue;
    for (int l = 0; l < 4; ++l)
        if (reinterpret_cast<uintptr_t>(w[l]) & 15u) return cudaErrorInvalidValue;
    if ((reinterpret_cast<uintptr_t>(x) & 15u) || (reinterpret_cast<uintptr_t>(y) & 15u) || ld_y % 4 ||
        (reinterpret_cast<uintptr_t>(bias[3]) & 15u))
        return cudaErrorInvalidValue;
    CUtensorMap mx, mw[4];
    const Mat X{x, M, in_dim, in_dim};
    const int din[4] = {in_dim, 256, 256, 256}, dout[4] = {256, 256, 256, out_dim};
    if (!make_map(&mx, X, M, in_dim, BM)) return cudaErrorInvalidValue;
    for (int l = 0; l < 4; ++l) {
        const Mat W{w[l], dout[l], din[l], din[l]};
        if (!make_map(&mw[l], W, dout[l], din[l], 256)) return cudaErrorInvalidValue;
    }
    cudaError_t e = fused_prepare();
    if (e != cudaSuccess) return e;
    FusedParams fp;
    for (int l = 0; l < 4; ++l) fp.bias[l] = bias[l];
    fp.y = y;
    fp.ld_y = ld_y;
    fp.M = (int)M;
    fp.in_dim = in_dim;
    fp.out_dim = out_dim;
    fp.err = err;
    fp.ring = fused_ring(in_dim);
    // fewer tiles than SMs: the output blocks of a tile go to several CTAs,
    // as many as leave no SM with a second unit
    const int tiles = (int)((M + BM - 1) / BM), n_ob = (out_dim + 255) / 256;
    fp.nsplit = std::max(1, std::min(n_ob, num_sms / tiles));
    const int units = tiles * fp.nsplit;
    const int grid = units < num_sms ? units : num_sms;
    return launch_chained(mlp_fused_forward_kernel, grid, kFThreads, fused_smem_bytes(in_dim), s, mx, mw[0], mw[1],
                          mw[2], mw[3], fp);
}

cudaError_t fused_prepare() {
    static int raised[64] = {};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 64 && raised[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(mlp_fused_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)std::max(fused_smem_bytes(192), fused_smem_bytes(256)));
    if (e == cudaSuccess && dev < 64) raised[dev] = 1;
    return e;
}

}  // namespace mlp
}  // namespace comet
