// bimanual_kernel.cu -- persistent evaluator of the bimanual variant: a box
// in the vertical plane flipped by two point hands on a ground contact
// (state x, z, theta, s_L, s_R; control twist, hand forces and sliding
// rates, ground force and centre of pressure; 507 modes = 3 ground x 13 x 13
// hand modes), one CTA of 128 threads per TO.
//
// The solver is the method of Sec. III-C with the Gauss-Newton model (the
// same steps as the pushing evaluator): PHR augmented Lagrangian, a
// backward sweep over w_k = (u_k, x_{k+1}) (17 x 17 S_k, Cholesky without
// pivoting, damping retries), trial steps alpha = 2^-i with the Armijo test,
// multiplier / penalty updates, the KKT stop test, and an FP64 certificate
// of v_hat (Eq. inexact_mode_value) and the KKT residual.
//
// Work per iteration:
//   A  a thread per stage: the 32 constraint rows and their Jacobians, one
//      after the other as straight code (each row's index a constant), the
//      multipliers, measures and the AL gradient; a stage's nonzeros go to the
//      CTA's workspace (L2-resident) as one packed record
//   M  a warp per two stages: the AL model over (u, x_{k+1}, x_k) in
//      registers, a model row per lane, from each row's nonzero pattern; the
//      12 u columns eliminated there (the pivot column through shared
//      memory); records to the workspace, in float4s
//   B  one warp, a row per lane: the sequential sweep eliminating the 5
//      x_{k+1} columns, the reduced blocks copied into shared memory ahead
//   gains and control steps stage-parallel, the forward chain on 5 lanes
//      from gains copied ahead
//   D  8 trial steps x stages over all threads, sums in shared memory
//   E  compensated state update
// Phase A used to run a lane per row: the warp then walked every row type's
// code for each stage (1,700 of a stage-iteration's 4,300 warp instructions),
// and phase M belonged to it, so that a trip that only updates multipliers
// built a model nobody used and a retry recomputed its rows.  With a thread
// per stage the rows cost 50 instructions per stage; 2,048 random orders of
// 1..6 segments took 213 -> 105 ms, the 507 one-segment orders 25 -> 15 ms.
// Then the sequential parts: a lane per row and copies ahead in B and the
// forward chain, two stages side by side and vector records in M: 105 -> 92
// ms and 15 -> 12.4 ms.  Results stayed the same to rounding: most orders bit
// for bit, isolated entries of mixed-length launches 1e-12 off.
//
// What bounds it (2,048 orders, cycles per TO-iteration with 4 CTAs on an
// SM): M 126 k, B 70 k, A 28 k, C 27 k, trials 23 k.  Issue slots are 27 %
// used: dependent chains (roots and reciprocals of 17 pivots per stage, one
// warp in B while three wait) and instruction fetches, not memory.

#include <cuda_runtime.h>
#include <cuda/annotated_ptr>
#include <math.h>
#include <stdint.h>

#include "comet.h"
#include "comet_internal.h"
#include "launch.h"

namespace comet {
namespace {

constexpr unsigned kFullB = 0xffffffffu;
constexpr int NX = 5, NU = 12, NR = 32, NL = 22, NWV = 17;
constexpr int NE = 23;               // elimination order (u 12, y 5, x 5, rhs)
constexpr int NRED = 11;             // reduced block (y 5, x 5, rhs)
constexpr int NTRI_RED = NRED * (NRED + 1) / 2;  // 66
// record layout (floats)
// Triangles are stored a row after the other, each row in whole float4s, so
// that a lane writes its row in one to three vector stores
__host__ __device__ constexpr int lrow(int i) { return i < 4 ? 4 * i : i < 8 ? 16 + 8 * (i - 4) : 48 + 12 * (i - 8); }
constexpr int R_LUU = 0;     // 96: u-block factor, lower triangle (12 rows)
constexpr int R_CPL = 96;    // 132: coupling rows (y, x, rhs) x 12 u columns
constexpr int R_RED = 228;   // 84: reduced (y, x, rhs) block (11 rows), its last float the u-block's PD flag
constexpr int R_PD = R_RED + lrow(10) + 11;
constexpr int R_YF = R_RED;  // 15 + 30 raw y-factor (+3 pad), then 30 gains, over the consumed block
static_assert(R_PD == R_RED + 83 && R_RED + 84 <= kBimRec, "record layout");
static_assert(R_YF % 4 == 0 && kBimRec % 4 == 0, "vector access to the raw factor");
// sweep copy ring: the reduced blocks, kBRing stages ahead
constexpr int kBSlot = 84, kBRing = 6;
constexpr int kCRing = 12;  // stages of gains in the same ring (forward chain)
static_assert(kCRing * 32 <= kBRing * kBSlot, "gains ring");

// stage Jacobian records (written by phase A, read by phase M): the entries of
// every row's pattern (bnz) one row after the other, a zero, and the local
// gradient in elimination order; chunk-major, float4 chunk q of stage k at
// 4 (q N_max + k), so that lanes over stages move whole lines
constexpr int NNZ = 85, J_ZERO = 85, J_GRAD = 88, J_REC = 112;
static_assert(J_REC <= kBimJac && J_REC % 4 == 0, "Jacobian record layout");
constexpr int NLAM = 33;  // multipliers per stage in shared memory: 32 and a pad (lanes over stages)

// local variables: x_k 0..4, u_k 5..16, x_{k+1} 17..21
enum { VX = 0, VZ, VTH, VSL, VSR, UXD, UZD, UTHD, UFNL, UFTL, USDL, UFNR, UFTR, USDR, ULN, ULT, UPC, VX1 };

__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }

// asynchronous global -> shared copies of 16 bytes with commit groups (the
// waits are hardware waits on the issuing thread's own groups)
__device__ __forceinline__ void bcp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void bcp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bcp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bcp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// reciprocal from the SFU (rcp.approx, about 1 ulp); the damped pivots are
// never subnormal
__device__ __forceinline__ float brcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// elimination position of local variable v; rhs = 22
__host__ __device__ constexpr int epos(int v) { return v >= 17 ? v - 5 : (v >= 5 ? v - 5 : v + 17); }
// local variable of elimination position e (e < 22)
__host__ __device__ constexpr int evar(int e) { return e < 17 ? e + 5 : e - 17; }


template <typename T>
struct BInst {
    T ax, az, mg, lbar, mu_g, mu_h, cg, ch, dt;
    T start[3], goal[3];
    T wT, wc, wf;  // control weights: wc (twist, sliding rates, p_c), wf (forces)
    int K;
};

// weight of control j (forces: f_n, f_t of both hands, lam_n, lam_t)
template <typename T>
__device__ __forceinline__ T rweight(const BInst<T>& P, int j) {
    return (j == 3 || j == 4 || j == 6 || j == 7 || j == 9 || j == 10) ? P.wf : P.wc;
}

template <typename T>
__device__ void load_inst(const DevInstance& d, BInst<T>& P) {
    const bool dbl = sizeof(T) == 8;
    P.ax = dbl ? (T)d.a_d[0] : (T)d.a[0];
    P.az = dbl ? (T)d.a_d[1] : (T)d.a[1];
    const T mass = dbl ? (T)d.mass_d : (T)d.mass;
    P.mg = mass * (T)9.81;
    P.lbar = P.ax > P.az ? P.ax : P.az;
    P.mu_g = dbl ? (T)d.ground_mu_d : (T)d.ground_mu;
    P.mu_h = dbl ? (T)d.mu_d : (T)d.mu;
    P.cg = sqrt(1 + P.mu_g * P.mu_g);
    P.ch = sqrt(1 + P.mu_h * P.mu_h);
    P.dt = dbl ? (T)d.dt_d : (T)d.dt;
    for (int i = 0; i < 3; ++i) {
        P.start[i] = dbl ? (T)d.start_d[i] : (T)d.start[i];
        P.goal[i] = dbl ? (T)d.goal_d[i] : (T)d.goal[i];
    }
    P.wT = dbl ? (T)d.w_terminal_d : (T)d.w_terminal;
    const T wc = dbl ? (T)d.w_control_d : (T)d.w_control;
    P.wc = wc;
    P.wf = wc / (P.mg * P.mg);
    P.K = d.K;
}

// per-stage quantities shared by the rows
template <typename T>
struct BStage {
    T cth, sth;
    int g, h[2];
    T n[2][2], t[2][2], a[2], ell[2];
    T Fwx, Fwz, tau;      // wrench sums (without gravity's force)
    T rcx, rcz, w, dw;    // pivot corner offset, support half-width
};

// Products and sums with their rounding written out (FP32): fm(a, b, c) is one
// fused multiply-add, m2(a, b) a product rounded by itself.  Left to the
// compiler, which of two products of a sum is fused depends on the code
// around it, and the rows are inlined in several phases.
__device__ __forceinline__ float fm(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fm(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ float m2(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double m2(double a, double b) { return a * b; }
__device__ __forceinline__ float a2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double a2(double a, double b) { return a + b; }

template <typename T>
__device__ __forceinline__ void stage_ctx(const BInst<T>& P, int mode, const T* x, const T* u, BStage<T>& S) {
    S.g = mode / 169;
    S.h[0] = (mode / 13) % 13;
    S.h[1] = mode % 13;
    const T th = x[VTH];
    if (sizeof(T) == 8) {
        double s, c;
        sincos((double)th, &s, &c);
        S.cth = (T)c;
        S.sth = (T)s;
    } else {
        float s, c;
        sincosf((float)th, &s, &c);
        S.cth = (T)c;
        S.sth = (T)s;
    }
    const T cth = S.cth, sth = S.sth;
    S.Fwx = u[ULT - 5];
    S.Fwz = u[ULN - 5];
    S.tau = fm(u[UPC - 5], u[ULN - 5], m2(x[VZ], u[ULT - 5]));
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int h = S.h[side];
        const int f = h == 0 ? 0 : (h - 1) / 3;
        const T nx = (f == 0) ? (T)1 : ((f == 2) ? (T)-1 : (T)0);
        const T nz = (f == 1) ? (T)1 : ((f == 3) ? (T)-1 : (T)0);
        S.n[side][0] = nx;
        S.n[side][1] = nz;
        S.t[side][0] = -nz;
        S.t[side][1] = nx;
        S.a[side] = (f % 2 == 0) ? P.ax : P.az;
        S.ell[side] = (f % 2 == 0) ? P.az : P.ax;
        if (h == 0) continue;
        const T fn = u[(side ? UFNR : UFNL) - 5], ft = u[(side ? UFTR : UFTL) - 5];
        const T s = x[side ? VSR : VSL];
        const T bx = fm(fn, nx, m2(ft, -nz)), bz = fm(fn, nz, m2(ft, nx));
        S.Fwx = a2(S.Fwx, fm(cth, bx, -m2(sth, bz)));
        S.Fwz = a2(S.Fwz, fm(sth, bx, m2(cth, bz)));
        S.tau = a2(S.tau, fm(-S.a[side], ft, -m2(s, fn)));
    }
    const T axc = m2(P.ax, cth), azs = m2(P.az, sth);
    S.rcx = a2(-axc, azs);
    S.rcz = fm(-P.ax, sth, -m2(P.az, cth));
    S.w = fm(axc, cth, m2(azs, sth));
    S.dw = m2(m2(2 * sth, cth), P.az - P.ax);
}

// hand rows of one side (q = 0..7): force, sliding rate and offset
__host__ __device__ constexpr int bnz_hand(bool right, int q, int a) {
    return (q == 0 || q == 3) ? (a == 0 ? (right ? UFNR : UFNL) : a == 1 ? (right ? UFTR : UFTL)
                                 : a == 2 ? (right ? USDR : USDL) : -1)
         : q == 1 ? (a == 0 ? (right ? UFTR : UFTL) : -1)
         : q == 2 ? (a == 0 ? (right ? USDR : USDL) : -1)
         : q == 4 ? (a == 0 ? (right ? UFNR : UFNL) : a == 1 ? (right ? UFTR : UFTL) : -1)
         : q == 5 ? (a == 0 ? (right ? UFNR : UFNL) : -1)
                  : (a == 0 ? (right ? VSR : VSL) : -1);
}

// Local variables that row r can depend on, over all modes (a superset of
// the nonzeros brow writes), ascending; -1 pads.  Kinematic rows: x_k,r,
// the rate and x_{k+1},r; wrench rows: the force components, the angle and
// (torque) z, the hands' offsets and the centre of pressure; ground rows:
// the twist, the ground force and p_c, the angle where the pivot enters;
// hand rows: that hand's force, sliding rate and offset.
__host__ __device__ constexpr int bnz(int r, int a) {
    return r < 5 ? (a == 0 ? r : a == 1 ? (r < 3 ? UXD + r : (r == 3 ? USDL : USDR)) : a == 2 ? VX1 + r : -1)
         : r == 5 ? (a == 0 ? VTH : a == 1 ? UFNL : a == 2 ? UFTL : a == 3 ? UFNR : a == 4 ? UFTR : a == 5 ? ULT : -1)
         : r == 6 ? (a == 0 ? VTH : a == 1 ? UFNL : a == 2 ? UFTL : a == 3 ? UFNR : a == 4 ? UFTR : a == 5 ? ULN : -1)
         : r == 7 ? (a == 0 ? VZ : a == 1 ? VSL : a == 2 ? VSR : a == 3 ? UFNL : a == 4 ? UFTL : a == 5 ? UFNR
                     : a == 6 ? UFTR : a == 7 ? ULN : a == 8 ? ULT : a == 9 ? UPC : -1)
         : r == 8 ? (a == 0 ? VTH : a == 1 ? UXD : a == 2 ? UZD : a == 3 ? UTHD : -1)
         : r == 9 ? (a == 0 ? VTH : a == 1 ? UZD : a == 2 ? UTHD : -1)
         : r == 10 ? (a == 0 ? VTH : a == 1 ? UTHD : a == 2 ? ULN : a == 3 ? ULT : a == 4 ? UPC : -1)
         : r == 11 ? (a == 0 ? UXD : a == 1 ? ULN : a == 2 ? ULT : -1)
         : r == 12 ? (a == 0 ? ULN : a == 1 ? ULT : -1)
         : r == 13 ? (a == 0 ? ULN : -1)
         : r <= 15 ? (a == 0 ? VTH : a == 1 ? UPC : -1)
         : bnz_hand(r >= 24, r - (r >= 24 ? 24 : 16), a);
}

// first entry of row r in the packed pattern (closed form: it has to fold to a
// constant where the rows are unrolled)
__host__ __device__ constexpr int bnz_first_hand(int q) {
    return q == 0 ? 0 : q == 1 ? 3 : q == 2 ? 4 : q == 3 ? 5 : q == 4 ? 8 : q == 5 ? 10 : q == 6 ? 11 : 12;
}
__host__ __device__ constexpr int bnz_first(int r) {
    return r < 5 ? 3 * r : r == 5 ? 15 : r == 6 ? 21 : r == 7 ? 27 : r == 8 ? 37 : r == 9 ? 41 : r == 10 ? 44
         : r == 11 ? 49 : r == 12 ? 52 : r == 13 ? 54 : r == 14 ? 55 : r == 15 ? 57
         : r < 24 ? 59 + bnz_first_hand(r - 16) : 72 + bnz_first_hand(r - 24);
}
constexpr bool bnz_first_ok() {
    int n = 0;
    for (int r = 0; r < NR; ++r) {
        if (bnz_first(r) != n) return false;
        for (int q = 0; q < 10 && bnz(r, q) >= 0; ++q) ++n;
    }
    return n == NNZ;
}
static_assert(bnz_first_ok(), "packed Jacobian offsets");

// Row r of an interval: scaled value c, presence, inequality flag, the
// physical factor (physical = c / scale) and, with WJ, the Jacobian over the
// 22 local variables.  dx = x_{k+1} - x_k (kinematic rows; computed from the
// compensated states by the caller).
template <typename T, bool WJ>
__device__ __forceinline__ void brow(int r, const BInst<T>& P, const BStage<T>& S, bool mL, bool mR, const T* x, const T* u,
                     const T* dx, T& c, T* J, bool& on, bool& ineq, T& scale) {
    // internally the force rows are divided by m g and the torque row by
    // m g l; scale maps a row back to physical units (physical = c / scale:
    // N, N m, W, m, m/s), as v_hat is scored (Sec. III-C "Stopping and
    // scoring")
    c = 0;
    on = true;
    ineq = (r >= 11 && r <= 15) || (r >= 19 && r <= 23) || (r >= 27);
    scale = 1;
    if (WJ)
        for (int j = 0; j < NL; ++j) J[j] = 0;
    const T mg = P.mg;
    if (r < 5) {
        const int vel = (r < 3) ? UXD + r : (r == 3 ? USDL : USDR);
        const T dxr = (r == 0) ? dx[0] : (r == 1) ? dx[1] : (r == 2) ? dx[2] : (r == 3) ? dx[3] : dx[4];
        const T ur = (r == 0) ? u[0] : (r == 1) ? u[1] : (r == 2) ? u[2] : (r == 3) ? u[USDL - 5] : u[USDR - 5];
        c = fm(-P.dt, ur, dxr);
        if (WJ) {
            J[r] = -1;
            J[VX1 + r] = 1;
            J[vel] = -P.dt;
        }
        if ((r == 3 && mL) || (r == 4 && mR)) on = false;
    } else if (r < 8) {
        const T sc = (r == 7) ? 1 / (mg * P.lbar) : 1 / mg;
        scale = sc;
        if (r == 5) c = m2(S.Fwx, sc);
        if (r == 6) c = m2(S.Fwz - mg, sc);
        if (r == 7) c = m2(S.tau, sc);
        if (WJ) {
            const T cth = S.cth, sth = S.sth;
            if (r == 5) J[ULT] = sc;
            if (r == 6) J[ULN] = sc;
            if (r == 7) {
                J[UPC] = u[ULN - 5] * sc;
                J[ULN] = u[UPC - 5] * sc;
                J[VZ] = u[ULT - 5] * sc;
                J[ULT] = x[VZ] * sc;
            }
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                if (S.h[side] == 0) continue;
                const int ufn = side ? UFNR : UFNL, uft = side ? UFTR : UFTL, vs = side ? VSR : VSL;
                const T nx = S.n[side][0], nz = S.n[side][1], tx = S.t[side][0], tz = S.t[side][1];
                const T fn = u[ufn - 5], ft = u[uft - 5];
                const T bx = fm(fn, nx, m2(ft, tx)), bz = fm(fn, nz, m2(ft, tz));
                const T wx = fm(cth, bx, -m2(sth, bz)), wz = fm(sth, bx, m2(cth, bz));
                if (r == 5) {
                    J[VTH] = fm(-wz, sc, J[VTH]);
                    J[ufn] = m2(fm(cth, nx, -m2(sth, nz)), sc);
                    J[uft] = m2(fm(cth, tx, -m2(sth, tz)), sc);
                } else if (r == 6) {
                    J[VTH] = fm(wx, sc, J[VTH]);
                    J[ufn] = m2(fm(sth, nx, m2(cth, nz)), sc);
                    J[uft] = m2(fm(sth, tx, m2(cth, tz)), sc);
                } else {
                    J[uft] = -S.a[side] * sc;
                    J[ufn] = -(side ? x[VSR] : x[VSL]) * sc;
                    J[vs] = -fn * sc;
                }
            }
        }
    } else if (r < 16) {
        const T xd = u[0], zd = u[1], thd = u[2], ln = u[ULN - 5], lt = u[ULT - 5], pc = u[UPC - 5];
        const T mu = P.mu_g;
        if (r == 8) {
            if (S.g == 0) {
                c = xd;
                if (WJ) J[UXD] = 1;
            } else if (S.g == 1) {
                c = zd;
                if (WJ) J[UZD] = 1;
            } else {
                c = fm(-thd, S.rcz, xd);
                if (WJ) {
                    J[UXD] = 1;
                    J[UTHD] = -S.rcz;
                    J[VTH] = -thd * S.rcx;
                }
            }
        } else if (r == 9) {
            if (S.g == 0) {
                c = zd;
                if (WJ) J[UZD] = 1;
            } else if (S.g == 1) {
                c = thd;
                if (WJ) J[UTHD] = 1;
            } else {
                c = fm(thd, S.rcx, zd);
                if (WJ) {
                    J[UZD] = 1;
                    J[UTHD] = S.rcx;
                    J[VTH] = -thd * S.rcz;
                }
            }
        } else if (r == 10) {
            if (S.g == 0) {
                c = thd;
                if (WJ) J[UTHD] = 1;
            } else if (S.g == 1) {
                const T s2 = 1 / (mg * mg);
                // factored, so that the difference near the edge is formed
                // before the product (no cancellation of two squares)
                c = m2(m2(fm(-mu, ln, lt), fm(mu, ln, lt)), s2);
                // physical: the friction force's distance from the cone
                // edge, |lam_t| - mu |lam_n| [N]
                const T den = fm(mu, fabs(ln), fabs(lt));
                scale = den > (T)0 ? den * s2 : (T)1;
                if (WJ) {
                    J[ULT] = 2 * lt * s2;
                    J[ULN] = -2 * mu * mu * ln * s2;
                }
            } else {
                c = pc - S.rcx;
                if (WJ) {
                    J[UPC] = 1;
                    J[VTH] = S.rcz;
                }
            }
        } else if (r == 11 || r == 12) {
            if (S.g != 1) {
                const T sc = 1 / (mg * P.cg), sg = (r == 11) ? (T)1 : (T)-1;
                scale = sc;
                c = m2(a2(sg * lt, -m2(mu, ln)), sc);
                if (WJ) {
                    J[ULT] = sg * sc;
                    J[ULN] = -mu * sc;
                }
            } else if (r == 11) {
                const T sc = 1 / mg;
                scale = sc;  // W
                c = m2(m2(lt, xd), sc);
                if (WJ) {
                    J[ULT] = xd * sc;
                    J[UXD] = lt * sc;
                }
            } else {
                on = false;
            }
        } else if (r == 13) {
            scale = 1 / mg;
            c = -ln / mg;
            if (WJ) J[ULN] = -1 / mg;
        } else {
            if (S.g == 2) {
                on = false;
            } else {
                const T sg = (r == 14) ? (T)1 : (T)-1;
                c = fm(sg, pc, -S.w);
                if (WJ) {
                    J[UPC] = sg;
                    J[VTH] = -S.dw;
                }
            }
        }
    } else {
        const bool side = r >= 24;
        const int q = r - (side ? 24 : 16);
        const int h = side ? S.h[1] : S.h[0];
        const int ufn = side ? UFNR : UFNL, uft = side ? UFTR : UFTL, usd = side ? USDR : USDL;
        const int vs = side ? VSR : VSL;
        const T fn = side ? u[UFNR - 5] : u[UFNL - 5], ft = side ? u[UFTR - 5] : u[UFTL - 5];
        const T sd = side ? u[USDR - 5] : u[USDL - 5], s = side ? x[VSR] : x[VSL];
        const T ell = side ? S.ell[1] : S.ell[0];
        if (h == 0) {
            if (q == 0) {
                scale = 1 / mg;
                c = fn / mg;
                if (WJ) J[ufn] = 1 / mg;
            } else if (q == 1) {
                scale = 1 / mg;
                c = ft / mg;
                if (WJ) J[uft] = 1 / mg;
            } else if (q == 2) {
                c = sd;
                if (WJ) J[usd] = 1;
            } else {
                on = false;
            }
        } else {
            const int kind = (h - 1) % 3;
            const T muh = P.mu_h, sch = 1 / (mg * P.ch);
            if (q == 1 || q == 2) {
                on = false;
            } else if (q == 0) {
                if (kind == 0) {
                    c = sd;
                    if (WJ) J[usd] = 1;
                } else {
                    const T sg = (kind == 1) ? (T)-1 : (T)1;
                    scale = sch;
                    c = m2(fm(sg * muh, fn, ft), sch);
                    if (WJ) {
                        J[uft] = sch;
                        J[ufn] = sg * muh * sch;
                    }
                }
            } else if (q == 3) {
                if (kind == 0) {
                    scale = sch;
                    c = m2(fm(-muh, fn, ft), sch);
                    if (WJ) {
                        J[uft] = sch;
                        J[ufn] = -muh * sch;
                    }
                } else {
                    const T sg = (kind == 1) ? (T)-1 : (T)1;
                    c = sg * sd;
                    if (WJ) J[usd] = sg;
                }
            } else if (q == 4) {
                if (kind == 0) {
                    scale = sch;
                    c = m2(fm(-muh, fn, -ft), sch);
                    if (WJ) {
                        J[uft] = -sch;
                        J[ufn] = -muh * sch;
                    }
                } else {
                    on = false;
                }
            } else if (q == 5) {
                scale = 1 / mg;
                c = -fn / mg;
                if (WJ) J[ufn] = -1 / mg;
            } else {
                const T sg = (q == 6) ? (T)1 : (T)-1;
                c = fm(sg, s, -ell);
                if (WJ) J[vs] = sg;
            }
        }
    }
    if (!on) {
        c = 0;
        if (WJ)
            for (int j = 0; j < NL; ++j) J[j] = 0;
    }
}

__device__ __forceinline__ float bwarp_max(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFullB, v, o));
    return v;
}
__device__ __forceinline__ float bwarp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullB, v, o);
    return v;
}

__device__ __forceinline__ void two_sum_b(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

struct BSmem {
    float *xh, *xl, *us, *lam, *dz, *gr;
    int* mi;     // per interval: mode | maskL << 10 | maskR << 11
    float* jbuf;          // per warp: two pairs of Jacobian records
    float* col;           // per warp: two pairs of pivot columns of 24
    uint16_t* at;         // [row][lane]: byte offset of the lane's entry in a record
    float* ring;          // sweep copy ring [kBRing][kBSlot] (16-byte aligned)
    float* red;           // reductions / broadcasts [64]
};

__host__ __device__ inline size_t bsmem_floats(int Nmax) {
    const size_t f = (size_t)10 * (Nmax + 1) + (size_t)NU * Nmax + 3 + (size_t)NLAM * Nmax +
                     2 * ((size_t)NWV * Nmax + NX) + (size_t)Nmax + 4 * (4 * J_REC + 96) + NR * 16 +
                     kBRing * kBSlot + 64;
    return (f + 3) / 4 * 4;
}

__device__ BSmem bcarve(float* p, int Nmax) {
    BSmem s;
    s.ring = p; p += kBRing * kBSlot;  // first: 16-byte aligned
    s.jbuf = p; p += 4 * 4 * J_REC;
    s.col = p; p += 4 * 96;
    s.at = reinterpret_cast<uint16_t*>(p); p += NR * 16;
    s.xh = p; p += NX * (Nmax + 1);
    s.xl = p; p += NX * (Nmax + 1);
    s.us = p; p += NU * Nmax;
    s.lam = p; p += 3 + NLAM * Nmax;
    s.dz = p; p += NWV * Nmax + NX;
    s.gr = p; p += NWV * Nmax + NX;
    s.mi = reinterpret_cast<int*>(p); p += Nmax;
    s.red = p;
    return s;
}

struct BCtx {
    const DevInstance* D;
    BInst<float> P;
    BSmem S;
    float* rec;
    float* jac;   // Jacobian records (chunk-major)
    int N, Np1, Nmax, len;
    int tid, warp, lane;
};

// compensated local variables of stage k at step alpha along dz
// (at alpha = 0 the step is not read: phase A runs before the first step of
// a TO exists, and its buffer also parks gradient parts during phase A)
__device__ __forceinline__ void load_stage(const BCtx& C, int k, float alpha, float* x, float* u, float* dx) {
    const int Np1 = C.Np1, N = C.N;
    const BSmem& S = C.S;
    const bool step = alpha != 0.f;
#pragma unroll
    for (int i = 0; i < NX; ++i) {
        const float h0 = S.xh[i * Np1 + k], h1 = S.xh[i * Np1 + k + 1];
        const float l0 = S.xl[i * Np1 + k] + (step ? alpha * S.dz[NWV * k + i] : 0.f);
        const float l1 = S.xl[i * Np1 + k + 1] + (step ? alpha * S.dz[NWV * (k + 1) + i] : 0.f);
        x[i] = h0 + l0;
        dx[i] = (h1 - h0) + (l1 - l0);
    }
#pragma unroll
    for (int j = 0; j < NU; ++j) u[j] = S.us[j * N + k] + (step ? alpha * S.dz[NWV * k + NX + j] : 0.f);
}

struct BMeasures {
    float viol, stat, comp;
    float vphys;  // violation in physical units (rows mapped back by c / scale)
    float cost;   // objective J at the iterate (scale of the stationarity test)
    bool finite;
};

// Phase A, a thread per stage: rows and their Jacobians (every row its own
// straight code, its index a constant), multipliers (PHR update at beta_old
// with `update`), the measures, the AL gradient into gr (x_{k+1} parts parked
// in dz) and the stage's Jacobian record for phase M.
__device__ BMeasures bphase_a(BCtx& C, float beta, bool update, float beta_old) {
    BSmem& S = C.S;
    const BInst<float>& P = C.P;
    const int N = C.N;
    float viol = 0.f, comp = 0.f, vph = 0.f, jc = 0.f;
    bool finite = true;
#pragma unroll 1
    for (int k = C.tid; k < N; k += kBimThreads) {
        float x[NX], u[NU], dx[NX];
        load_stage(C, k, 0.f, x, u, dx);
        const int mi = S.mi[k];
        BStage<float> St;
        stage_ctx(P, mi & 1023, x, u, St);
        float* lam = S.lam + 3 + NLAM * k;
        cuda::annotated_ptr<float4, cuda::access_property::persisting> jac(reinterpret_cast<float4*>(C.jac) + k);
        float g[NL], out[J_REC];
#pragma unroll
        for (int j = 0; j < NL; ++j) g[j] = 0.f;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float c, sc, J[NL];
            bool on, iq;
            brow<float, true>(r, P, St, (mi >> 10) & 1, (mi >> 11) & 1, x, u, dx, c, J, on, iq, sc);
            float l = lam[r];
            if (update && on) {
                const float t = fm(beta_old, c, l);
                l = iq ? fmaxf(t, 0.f) : t;
                lam[r] = l;
            }
            const float t = fm(beta, c, l);
            const bool act = on && (!iq || t > 0.f);
            const float y = act ? (iq ? fmaxf(t, 0.f) : t) : 0.f;
            if (on) {
                const float vr = iq ? fmaxf(c, 0.f) : fabsf(c);
                viol = fmaxf(viol, vr);
                vph = fmaxf(vph, vr / sc);
                if (iq) comp = fmaxf(comp, fabsf(y * c));
                if (!isfinite(c)) finite = false;
            }
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                const int v = bnz(r, q);
                if (v < 0) break;
                const float a = act ? J[v] : 0.f;
                out[bnz_first(r) + q] = a;
                g[v] = fm(y, a, g[v]);
            }
        }
#pragma unroll
        for (int j = 0; j < NU; ++j) g[NX + j] = fm(2.f * rweight(P, j), S.us[j * N + k], g[NX + j]);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            if (j < NWV)
                S.gr[NWV * k + j] = g[j];
            else
                S.dz[NWV * (k + 1) + j - NWV] = g[j];
        }
#pragma unroll
        for (int i = NNZ; i < J_GRAD; ++i) out[i] = 0.f;
#pragma unroll
        for (int e = 0; e < NL; ++e) out[J_GRAD + e] = g[evar(e)];
        out[J_GRAD + NL] = out[J_GRAD + NL + 1] = 0.f;
#pragma unroll
        for (int q = 0; q < J_REC / 4; ++q)
            jac[(int64_t)q * C.Nmax] = make_float4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
    }
    // the cost's control terms: four chains over the stages (k mod 4), on the
    // warp with the fewest stages
    if (C.warp == 3 && C.lane < 4) {
#pragma unroll 1
        for (int k = C.lane; k < N; k += 4) {
#pragma unroll
            for (int j = 0; j < NU; ++j) {
                const float uj = S.us[j * N + k];
                jc = fm(m2(rweight(P, j), uj), uj, jc);
            }
        }
    }
    __syncthreads();
    // initial pose rows and the combined gradient
    const int tid = C.tid, Np1 = C.Np1;
    float stat = 0.f;
    if (tid < 3) {
        float l = S.lam[tid];
        const float c = (S.xh[tid * Np1] - P.start[tid]) + S.xl[tid * Np1];
        if (update) {
            l = l + beta_old * c;
            S.lam[tid] = l;
        }
        viol = fmaxf(viol, fabsf(c));
        vph = fmaxf(vph, fabsf(c));
        if (!isfinite(c)) finite = false;
    }
    if (tid == 96)
        for (int i = 0; i < 3; ++i) {
            const float e = (S.xh[i * Np1 + N] - P.goal[i]) + S.xl[i * Np1 + N];
            jc = fm(m2(P.wT, e), e, jc);
        }
    __syncthreads();
    for (int k = tid; k <= N; k += kBimThreads) {
        for (int i = 0; i < NX; ++i) {
            float g = (k < N) ? S.gr[NWV * k + i] : 0.f;
            if (k > 0) g += S.dz[NWV * k + i];
            if (k == N && i < 3) g += 2.f * P.wT * ((S.xh[i * Np1 + N] - P.goal[i]) + S.xl[i * Np1 + N]);
            if (k == 0 && i < 3) g += S.lam[i] + beta * ((S.xh[i * Np1] - P.start[i]) + S.xl[i * Np1]);
            S.gr[NWV * k + i] = g;
            stat = fmaxf(stat, fabsf(g));
            if (!isfinite(g)) finite = false;
        }
        if (k < N)
            for (int j = 0; j < NU; ++j) {
                const float g = S.gr[NWV * k + NX + j];
                stat = fmaxf(stat, fabsf(g));
                if (!isfinite(g)) finite = false;
            }
    }
    // block reductions
    viol = bwarp_max(viol);
    stat = bwarp_max(stat);
    comp = bwarp_max(comp);
    vph = bwarp_max(vph);
    const bool fin = __all_sync(kFullB, finite);
    __syncthreads();
    if (C.lane == 0) {
        S.red[C.warp] = viol;
        S.red[4 + C.warp] = stat;
        S.red[8 + C.warp] = comp;
        S.red[12 + C.warp] = fin ? 1.f : 0.f;
        S.red[24 + C.warp] = vph;
    }
    if (C.warp == 3 && C.lane < 4) S.red[28 + C.lane] = jc;
    __syncthreads();
    BMeasures m;
    m.viol = fmaxf(fmaxf(S.red[0], S.red[1]), fmaxf(S.red[2], S.red[3]));
    m.stat = fmaxf(fmaxf(S.red[4], S.red[5]), fmaxf(S.red[6], S.red[7]));
    m.comp = fmaxf(fmaxf(S.red[8], S.red[9]), fmaxf(S.red[10], S.red[11]));
    m.finite = S.red[12] > 0.f && S.red[13] > 0.f && S.red[14] > 0.f && S.red[15] > 0.f;
    m.vphys = fmaxf(fmaxf(S.red[24], S.red[25]), fmaxf(S.red[26], S.red[27]));
    m.cost = (S.red[28] + S.red[29]) + (S.red[30] + S.red[31]);
    __syncthreads();
    return m;
}

// Phase M, a warp per two stages: the AL model over (u, x_{k+1}, x_k) from the
// stage's Jacobian record and the elimination of the 12 u columns, a model row
// per lane in registers; records for the sweep, the gains and the controls.
// The next two records are copied into shared memory meanwhile.
__device__ void bphase_m(BCtx& C, float beta, float rho) {
    BSmem& S = C.S;
    const BInst<float>& P = C.P;
    const int N = C.N, lane = C.lane, warp = C.warp;
    float* jb = S.jbuf + warp * 4 * J_REC;
    float* colb = S.col + warp * 96;
    auto fetch = [&](int k, int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (k + 4 * h < N && lane < J_REC / 4)
                bcp_async16(jb + (2 * buf + h) * J_REC + 4 * lane, C.jac + 4 * ((int64_t)lane * C.Nmax + k + 4 * h));
        bcp_async_commit();
    };
    fetch(warp, 0);
    int buf = 0;
    // Stages k and k + 4 side by side: a pivot is a chain of a shuffle, a
    // square root, a division and a trip through shared memory (about 250
    // cycles), which the other stage shares.  Six-segment orders, 64 of them /
    // 2,048 of mixed length: one stage at a time 92 k / 139 k cycles per
    // iteration, two with roots of their own 96 k / 158 k (the slow paths of
    // the exact root and division keep the chains apart), with one root for
    // both and vector records 70 k / 126 k.  A last stage without a partner
    // is done twice.
#pragma unroll 1
    for (int k = warp; k < N; k += 8, buf ^= 1) {
        fetch(k + 8, buf ^ 1);
        bcp_async_wait<1>();
        __syncwarp();
        const bool two = k + 4 < N;
        const float* J0 = jb + 2 * buf * J_REC;
        const float* Js[2] = {J0, two ? J0 + J_REC : J0};
        // lane i < 22 holds row i of the lower triangle over (u, y, x) in
        // elimination order (and lane 22 the rhs row).  Row i = sum_r J_r[v_i]
        // J_r over the active rows in row order; for row r only the columns of
        // its pattern (bnz) are added, the others being exact zeros: the
        // lane's own entry times a broadcast Jacobian value
        float row[2][NE];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int cc = 0; cc < NE; ++cc) row[h][cc] = 0.f;
        float4 t4[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int at = S.at[32 * r + lane];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float a = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(Js[h]) + at);
#pragma unroll
                for (int q = 0; q < 10; ++q) {
                    if (bnz(r, q) < 0) break;
                    const int n = bnz_first(r) + q;
                    if (n % 4 == 0) t4[h] = *reinterpret_cast<const float4*>(Js[h] + n);
                    const float b = n % 4 == 0 ? t4[h].x : n % 4 == 1 ? t4[h].y : n % 4 == 2 ? t4[h].z : t4[h].w;
                    // a row of one entry is added as a rounded product
                    float& m = row[h][epos(bnz(r, q))];
                    m = bnz(r, 1) < 0 ? a2(m, m2(a, b)) : fm(a, b, m);
                }
            }
        }
        // beta, then the cost and damping on the diagonal (u: cost + rho,
        // x_{k+1}: rho); the gradient as the rhs row (lane 22)
#pragma unroll
        for (int cc = 0; cc < NE - 1; ++cc) {
            const float dg = cc < 12 ? fm(2.f, rweight(P, cc), rho) : rho;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                row[h][cc] = m2(row[h][cc], beta);
                if (lane == cc && cc < 17) row[h][cc] = a2(row[h][cc], dg);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const float4 t = *reinterpret_cast<const float4*>(Js[h] + J_GRAD + 4 * q);
                if (lane == NE - 1) {
                    row[h][4 * q] = t.x;
                    row[h][4 * q + 1] = t.y;
                    if (4 * q + 2 < NE - 1) {
                        row[h][4 * q + 2] = t.z;
                        row[h][4 * q + 3] = t.w;
                    }
                }
            }
        // eliminate the u block (12 Cholesky columns): lane i < 23 holds row i
        // of the lower triangle (entries 0..i; what the updates leave above the
        // diagonal is never read).  The scaled column goes through shared
        // memory (two buffers, one warp barrier per pivot) and comes back as
        // broadcasts, four entries a load.  A non-positive pivot marks the record.
        bool pd[2] = {true, true};
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            float* col = colb + 48 * (j & 1);
            // the lower half-warp takes stage k's pivot, the upper one k + 4's,
            // so that both roots and reciprocals cost one pass
            const float d0 = __shfl_sync(kFullB, row[0][j], j), d1 = __shfl_sync(kFullB, row[1][j], j);
            pd[0] = pd[0] && (d0 > 0.f);
            pd[1] = pd[1] && (d1 > 0.f);
            const float l = sqrtf(fmaxf(lane < 16 ? d0 : d1, 1e-30f));
            const float il = 1.f / l;
            const float lx = __shfl_xor_sync(kFullB, l, 16), ilx = __shfl_xor_sync(kFullB, il, 16);
            row[0][j] = lane == j ? l : m2(row[0][j], lane < 16 ? il : ilx);  // j < 16: l is the lane's own
            row[1][j] = lane == j ? lx : m2(row[1][j], lane < 16 ? ilx : il);
            if (lane < 24) {
                col[lane] = row[0][j];
                col[24 + lane] = row[1][j];
            }
            __syncwarp();
#pragma unroll
            for (int q = (j + 1) / 4; q < 6; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 t = *reinterpret_cast<const float4*>(col + 24 * h + 4 * q);
                    const float b[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (4 * q + i > j && 4 * q + i < NE)
                            row[h][4 * q + i] = fm(-row[h][j], b[i], row[h][4 * q + i]);
                }
        }
        // records from the rows: the u factor (rows 0..11), the coupling
        // rows (12..22) x u columns, the reduced (y, x, rhs) block
        // record stores with the persisting (evict-last) L2 priority: the
        // CTAs' workspaces fit in L2 and are rewritten every iteration
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && !two) break;
            float* rk = C.rec + (size_t)(k + 4 * h) * kBimRec;
            const float* w = row[h];
            if (lane < NE) {
                cuda::annotated_ptr<float4, cuda::access_property::persisting> rec(
                    reinterpret_cast<float4*>(rk + (lane < 12 ? R_LUU + lrow(lane) : R_CPL + 12 * (lane - 12))));
                rec[0] = make_float4(w[0], w[1], w[2], w[3]);
                if (lane >= 4) rec[1] = make_float4(w[4], w[5], w[6], w[7]);
                if (lane >= 8) rec[2] = make_float4(w[8], w[9], w[10], w[11]);
            }
            if (lane >= 12 && lane < NE) {
                cuda::annotated_ptr<float4, cuda::access_property::persisting> rec(
                    reinterpret_cast<float4*>(rk + R_RED + lrow(lane - 12)));
                rec[0] = make_float4(w[12], w[13], w[14], w[15]);
                if (lane >= 16) rec[1] = make_float4(w[16], w[17], w[18], w[19]);
                if (lane >= 20) rec[2] = make_float4(w[20], w[21], w[22], pd[h] ? 1.f : -1.f);
            }
        }
        __syncwarp();
    }
    bcp_async_wait_all();
    __syncthreads();
}

// Sweep over k = N-1 .. 0 on warp 0, a lane per row of the reduced 11 x 11
// lower triangle (y 0..4, x 0..4, rhs; the lanes above repeat the rhs row).
// The block arrives from the record through a cp.async ring kBRing stages
// ahead.  V_{k+1} and v_{k+1} are the rows 5.. of the stage before: a shuffle
// of five values moves V to the y rows, v stays in the rhs lane.  Per pivot
// the lanes take the raw pivot column by shuffles while the SFU reciprocal of
// the pivot is under way; a lane writes its row's raw y-factor entries (15 y-y
// entries, then the (x, rhs) rows) for the gains.  Every lane running the
// whole stage (330 instructions, about 1,100 cycles) took 57 k cycles per
// iteration on 64 six-segment orders and 78 k on 2,048 mixed ones, this takes
// 56 k and 70 k.  Then the x_0 block; publishes the
// factorisation status to all threads and dx0 into red[16..20].
__device__ bool bphase_b(BCtx& C, float beta, float rho) {
    BSmem& S = C.S;
    const BInst<float>& P = C.P;
    const int N = C.N, Np1 = C.Np1, lane = C.lane;
    if (C.warp == 0) {
        const int row = min(lane, 10), at0 = lrow(row);
        // rows 5.. of "stage N": the terminal cost's V_N (lanes 5..9), v_N (lane 10)
        float m[11];
#pragma unroll
        for (int l = 0; l < 11; ++l) m[l] = 0.f;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (lane == 5 + l) m[5 + l] = 2.f * P.wT;
            if (row == 10) m[5 + l] = 2.f * P.wT * ((S.xh[l * Np1 + N] - P.goal[l]) + S.xl[l * Np1 + N]);
        }
#pragma unroll
        for (int d = 0; d < kBRing; ++d) {
            const int kk = N - 1 - d;
            if (kk >= 0 && lane < kBSlot / 4)
                bcp_async16(S.ring + d * kBSlot + 4 * lane, C.rec + (size_t)kk * kBimRec + R_RED + 4 * lane);
            bcp_async_commit();
        }
        bool ok = true;
        int slot = kBRing - 1;  // ring slot of stage k: (N - 1 - k) mod kBRing
        // where the lane's y-factor entries go: row i < 5 its entries 0..i, the
        // others five entries each
        const int out0 = R_YF + (row < 5 ? row * (row + 1) / 2 : 15 + 5 * (row - 5));
#pragma unroll 1
        for (int k = N - 1; k >= 0; --k) {
            slot = (slot == kBRing - 1) ? 0 : slot + 1;
            bcp_async_wait<kBRing - 1>();
            __syncwarp();
            const float* sl = S.ring + slot * kBSlot;
            bool pd = sl[R_PD - R_RED] > 0.f;
            float V[5];
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                const float t = __shfl_sync(kFullB, m[5 + l], (lane + 5) & 31);
                V[l] = row == 10 ? m[5 + l] : t;
            }
            // entries past the row's own are never used (they stay inside the slot)
#pragma unroll
            for (int l = 0; l < 11; ++l) m[l] = sl[at0 + l];
            __syncwarp();
            {
                const int kk = k - kBRing;
                if (kk >= 0 && lane < kBSlot / 4)
                    bcp_async16(S.ring + slot * kBSlot + 4 * lane, C.rec + (size_t)kk * kBimRec + R_RED + 4 * lane);
                bcp_async_commit();
            }
#pragma unroll
            for (int l = 0; l < 5; ++l)
                if (row < 5 || row == 10) m[l] = a2(m[l], V[l]);
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const float p = __shfl_sync(kFullB, m[j], j);
                float c[11];
#pragma unroll
                for (int l = j + 1; l < 11; ++l) c[l] = __shfl_sync(kFullB, m[j], l);
                pd = pd && (p > 0.f);
                const float a = m2(m[j], brcp_approx(p));
                if (row > j) {
#pragma unroll
                    for (int l = j + 1; l < 11; ++l) m[l] = fm(-a, c[l], m[l]);
                }
            }
            if (!pd) {  // the same on every lane
                ok = false;
                break;
            }
            if (lane < 11) {
                cuda::annotated_ptr<float, cuda::access_property::persisting> o(C.rec + (size_t)k * kBimRec + out0);
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (row >= 5 || j <= row) o[j] = m[j];
            }
        }
        // V_0, v_0 to every lane
        float V[15], v[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
#pragma unroll
            for (int j = 0; j <= i; ++j) V[tri(i, j)] = __shfl_sync(kFullB, m[5 + j], 5 + i);
            v[i] = __shfl_sync(kFullB, m[5 + i], 10);
        }
        bcp_async_wait_all();
        __syncwarp();
        // x_0 block (every lane), Cholesky with reciprocal pivots
        bool pd0 = ok;
        float d0[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        if (ok) {
            float H[5][5], g[5], L[5][5], il[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
#pragma unroll
                for (int j = 0; j < 5; ++j) H[i][j] = V[i >= j ? tri(i, j) : tri(j, i)];
                H[i][i] += rho;
                g[i] = v[i];
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                H[i][i] += beta;
                g[i] += S.lam[i] + beta * ((S.xh[i * Np1] - P.start[i]) + S.xl[i * Np1]);
            }
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                float d = H[j][j];
#pragma unroll
                for (int q = 0; q < j; ++q) d -= L[j][q] * L[j][q];
                pd0 = pd0 && d > 0.f;
                il[j] = rsqrtf(fmaxf(d, 1e-30f));
#pragma unroll
                for (int i = j + 1; i < 5; ++i) {
                    float s = H[i][j];
#pragma unroll
                    for (int q = 0; q < j; ++q) s -= L[i][q] * L[j][q];
                    L[i][j] = s * il[j];
                }
            }
            float yv[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                float s = g[i];
#pragma unroll
                for (int q = 0; q < i; ++q) s -= L[i][q] * yv[q];
                yv[i] = s * il[i];
            }
#pragma unroll
            for (int i = 4; i >= 0; --i) {
                float s = yv[i];
#pragma unroll
                for (int q = i + 1; q < 5; ++q) s -= L[q][i] * d0[q];
                d0[i] = s * il[i];
            }
        }
        if (lane == 0) {
            if (ok)
                for (int i = 0; i < 5; ++i) S.red[16 + i] = -d0[i];
            S.red[21] = pd0 ? 1.f : 0.f;
        }
    }
    __syncthreads();
    const bool res = S.red[21] > 0.f;
    __syncthreads();
    return res;
}

// gains K_y = -L_y^{-T} [l_{x,y} | l_{rhs,y}] (5 x 6) per stage
__device__ void bphase_gains(BCtx& C) {
#pragma unroll 1
    for (int k = C.tid; k < C.N; k += kBimThreads) {
        float* rec = C.rec + (size_t)k * kBimRec;
        // raw factor: 15 y-y entries, then the (x, rhs) rows, as vector loads
        float m[48];
        const float4* r4 = reinterpret_cast<const float4*>(rec + R_YF);
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            const float4 t = r4[q];
            m[4 * q] = t.x;
            m[4 * q + 1] = t.y;
            m[4 * q + 2] = t.z;
            m[4 * q + 3] = t.w;
        }
        float ly[5][5], il[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            il[j] = rsqrtf(m[tri(j, j)]);
#pragma unroll
            for (int i = j + 1; i < 5; ++i) ly[i][j] = m[tri(i, j)] * il[j];
#pragma unroll
            for (int c = 0; c < 6; ++c) m[15 + 5 * c + j] *= il[j];
        }
        // K (row i at R_YF + 6 i), two pad floats, as vector stores
        float o[32];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
#pragma unroll
            for (int i = 4; i >= 0; --i) {
                float s = -m[15 + 5 * c + i];
#pragma unroll
                for (int q = i + 1; q < 5; ++q) s -= ly[q][i] * o[6 * q + c];
                o[6 * i + c] = s * il[i];
            }
        }
        o[30] = o[31] = 0.f;
        cuda::annotated_ptr<float4, cuda::access_property::persisting> w4(reinterpret_cast<float4*>(rec + R_YF));
#pragma unroll
        for (int q = 0; q < 8; ++q) w4[q] = make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
    }
    __syncthreads();
}

// forward pass: the chain on 5 lanes of warp 0, then the control steps;
// returns D = grad . dz
__device__ float bphase_c(BCtx& C) {
    BSmem& S = C.S;
    const int N = C.N;
    if (C.warp == 0) {
        float dxi = (C.lane < 5) ? S.red[16 + C.lane] : 0.f;
        if (C.lane < 5) S.dz[C.lane] = dxi;
        float dxv[5];
        #pragma unroll
        for (int i = 0; i < 5; ++i) dxv[i] = __shfl_sync(kFullB, dxi, i);
        // the gains arrive through a copy ring kCRing stages ahead (a stage's
        // 32 floats per slot); read from the workspace one stage at a time,
        // the chain waited for the L2 at every stage (gains, chain and control
        // steps together 44 k cycles per iteration of 2,048 orders, now 27 k)
        auto fetch = [&](int k) {
            if (k < N && C.lane < 8)
                bcp_async16(S.ring + (k % kCRing) * 32 + 4 * C.lane, C.rec + (size_t)k * kBimRec + R_YF + 4 * C.lane);
            bcp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < kCRing; ++k) fetch(k);
        const int gl = C.lane < 5 ? 6 * C.lane : 0;
#pragma unroll 1
        for (int k = 0; k < N; ++k) {
            bcp_async_wait<kCRing - 1>();
            __syncwarp();
            const float* g = S.ring + (k % kCRing) * 32 + gl;
            float gv[6];
            #pragma unroll
            for (int j = 0; j < 6; ++j) gv[j] = g[j];
            __syncwarp();
            fetch(k + kCRing);
            float w = gv[5];
            #pragma unroll
            for (int j = 0; j < 5; ++j) w = fm(gv[j], dxv[j], w);
            if (C.lane < 5) S.dz[NWV * (k + 1) + C.lane] = w;
            #pragma unroll
            for (int i = 0; i < 5; ++i) dxv[i] = __shfl_sync(kFullB, w, i);
        }
        bcp_async_wait_all();
        __syncwarp();
    }
    __syncthreads();
#pragma unroll 1
    for (int k = C.tid; k < N; k += kBimThreads) {
        const float* rec = C.rec + (size_t)k * kBimRec;
        float xa[5], xb[5];
        #pragma unroll
        for (int i = 0; i < 5; ++i) {
            xa[i] = S.dz[NWV * k + i];
            xb[i] = S.dz[NWV * (k + 1) + i];
        }
        // R = l_rhs + l_y dx_{k+1} + l_x dx_k over the u columns, then
        // L^T du = -R; the record's rows as vector loads
        auto vec = [&](int at, int q) { return *reinterpret_cast<const float4*>(rec + at + 4 * q); };
        float R[NU];
        #pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 t = vec(R_CPL + 12 * 10, q);
            R[4 * q] = t.x, R[4 * q + 1] = t.y, R[4 * q + 2] = t.z, R[4 * q + 3] = t.w;
        }
        #pragma unroll
        for (int i = 0; i < 5; ++i)
            #pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float4 y = vec(R_CPL + 12 * i, q), x = vec(R_CPL + 12 * (5 + i), q);
                const float yv[4] = {y.x, y.y, y.z, y.w}, xv[4] = {x.x, x.y, x.z, x.w};
                #pragma unroll
                for (int e = 0; e < 4; ++e)
                    R[4 * q + e] = a2(R[4 * q + e], fm(yv[e], xb[i], m2(xv[e], xa[i])));
            }
        float L[78];
        #pragma unroll
        for (int i = 0; i < NU; ++i)
            #pragma unroll
            for (int q = 0; q <= i / 4; ++q) {
                const float4 t = vec(R_LUU + lrow(i), q);
                const float v[4] = {t.x, t.y, t.z, t.w};
                #pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (4 * q + e <= i) L[tri(i, 4 * q + e)] = v[e];
            }
        float du[NU];
        #pragma unroll
        for (int j = NU - 1; j >= 0; --j) {
            float s = -R[j];
            #pragma unroll
            for (int i = j + 1; i < NU; ++i) s = fm(-L[tri(i, j)], du[i], s);
            du[j] = s / L[tri(j, j)];
        }
        #pragma unroll
        for (int j = 0; j < NU; ++j) S.dz[NWV * k + NX + j] = du[j];
    }
    __syncthreads();
    float D = 0.f;
    for (int t = C.tid; t < NWV * N + NX; t += kBimThreads) D += S.gr[t] * S.dz[t];
    D = bwarp_sum(D);
    if (C.lane == 0) S.red[24 + C.warp] = D;
    __syncthreads();
    const float Dt = S.red[24] + S.red[25] + S.red[26] + S.red[27];
    __syncthreads();
    return Dt;
}

__device__ __forceinline__ float brow_al(bool ineq, float lam, float beta, float inv2b, float c) {
    if (!ineq) return fm(lam, c, m2(m2(m2(0.5f, beta), c), c));
    const float t = fmaxf(fm(beta, c, lam), 0.f);
    return m2(fm(t, t, -m2(lam, lam)), inv2b);
}

// trial merits for alpha in {0, 1, ..., 2^-6}; returns the accepted alpha
__device__ float bphase_d(BCtx& C, float beta, float D, const SolverParams& sp) {
    BSmem& S = C.S;
    const BInst<float>& P = C.P;
    const int N = C.N, Np1 = C.Np1;
    // Trials four at a time (thread = trial + 4 x stage group, 32 groups),
    // largest alpha first: {1/8 .. 1/64} only when none of {1, 1/2, 1/4}
    // passes, which leaves the accepted alpha (the largest passing) unchanged.
    const int sub = C.tid & 3, grp = C.tid >> 2;
    const float inv2b = 0.5f / beta;
    float phi0 = 0.f, slack = 0.f, acc = 0.f;
#pragma unroll 1
    for (int batch = 0; batch < 2; ++batch) {
        if (batch == 1 && sp.n_alpha < 4) break;
        const int a = 4 * batch + sub;
        const float alpha = (a == 0) ? 0.f : ldexpf(1.f, -(a - 1));
        float phi = 0.f;
        if (a <= sp.n_alpha) {
#pragma unroll 1
            for (int k = grp; k < N; k += 32) {
                float x[NX], u[NU], dx[NX];
                load_stage(C, k, alpha, x, u, dx);
                const int mi = S.mi[k];
                BStage<float> St;
                stage_ctx(P, mi & 1023, x, u, St);
                const float* lam = S.lam + 3 + NLAM * k;
#pragma unroll
                for (int j = 0; j < NU; ++j) phi = fm(m2(rweight(P, j), u[j]), u[j], phi);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    float c, sc;
                    bool on, iq;
                    brow<float, false>(r, P, St, (mi >> 10) & 1, (mi >> 11) & 1, x, u, dx, c, nullptr, on, iq, sc);
                    if (on) phi = a2(phi, brow_al(iq, lam[r], beta, inv2b, c));
                }
                if (k == 0)
                    for (int i = 0; i < 3; ++i) {
                        const float c = (S.xh[i * Np1] - P.start[i]) + (S.xl[i * Np1] + alpha * S.dz[i]);
                        phi = a2(phi, brow_al(false, S.lam[i], beta, inv2b, c));
                    }
                if (k == N - 1)
                    for (int i = 0; i < 3; ++i) {
                        const float e =
                            (S.xh[i * Np1 + N] - P.goal[i]) + (S.xl[i * Np1 + N] + alpha * S.dz[NWV * N + i]);
                        phi = fm(m2(P.wT, e), e, phi);
                    }
            }
        }
        // threads with the same trial: xor 4, 8, 16 inside the warp, then the warps
        phi += __shfl_xor_sync(kFullB, phi, 4);
        phi += __shfl_xor_sync(kFullB, phi, 8);
        phi += __shfl_xor_sync(kFullB, phi, 16);
        if (C.lane < 4) S.red[32 + C.warp * 4 + C.lane] = phi;
        __syncthreads();
        if (C.tid == 0) {
            float ph[4];
            for (int q = 0; q < 4; ++q) ph[q] = S.red[32 + q] + S.red[36 + q] + S.red[40 + q] + S.red[44 + q];
            if (batch == 0) {
                phi0 = ph[0];
                slack = sp.ls_slack * fabsf(phi0);
            }
            const bool flat = fabsf(D) <= slack;
            float take = 0.f;
            for (int q = (batch == 0) ? 1 : 0; q < 4; ++q) {
                const int aq = 4 * batch + q;
                if (aq > sp.n_alpha) break;
                const float al = ldexpf(1.f, -(aq - 1));
                if (ph[q] <= phi0 + sp.armijo_c1 * al * D || (aq == 1 && flat && ph[q] <= phi0 + slack)) {
                    take = al;
                    break;
                }
            }
            S.red[30] = take;
        }
        __syncthreads();
        acc = S.red[30];
        __syncthreads();
        if (acc > 0.f) break;
    }
    return acc;
}

__device__ void bphase_e(BCtx& C, float alpha) {
    BSmem& S = C.S;
    const int N = C.N, Np1 = C.Np1;
    for (int t = C.tid; t < NX * Np1; t += kBimThreads) {
        const int i = t / Np1, k = t - i * Np1;
        float s, e;
        two_sum_b(S.xh[t], S.xl[t] + alpha * S.dz[NWV * k + i], s, e);
        S.xh[t] = s;
        S.xl[t] = e;
    }
    for (int t = C.tid; t < NU * N; t += kBimThreads) {
        const int j = t / N, k = t - j * N;
        S.us[t] += alpha * S.dz[NWV * k + NX + j];
    }
    __syncthreads();
}

// FP64 certificate: cost, physical violation, KKT residual (stationarity
// with the multiplier estimates at beta); scratch doubles in the workspace
struct BCert {
    double cost, viol, stat;
    bool finite;
};

__device__ BCert bcertify(BCtx& C, float beta_f) {
    BSmem& S = C.S;
    const int N = C.N, Np1 = C.Np1;
    BInst<double> P;
    load_inst(*C.D, P);
    const double beta = beta_f;
    double* g64 = reinterpret_cast<double*>(C.rec);  // [17 N + 5] then [5 (N + 1)]
    double* g64b = g64 + (NWV * N + NX);
    double cost = 0.0, viol = 0.0;
    bool finite = true;
    for (int k = C.tid; k < N; k += kBimThreads) {
        double x[NX], u[NU], dx[NX];
        for (int i = 0; i < NX; ++i) {
            const double a0 = (double)S.xh[i * Np1 + k] + (double)S.xl[i * Np1 + k];
            const double a1 = (double)S.xh[i * Np1 + k + 1] + (double)S.xl[i * Np1 + k + 1];
            x[i] = a0;
            dx[i] = a1 - a0;
        }
        for (int j = 0; j < NU; ++j) u[j] = (double)S.us[j * N + k];
        const int mi = S.mi[k];
        BStage<double> St;
        stage_ctx(P, mi & 1023, x, u, St);
        double g[NL];
        for (int j = 0; j < NL; ++j) g[j] = 0.0;
        for (int j = 0; j < NU; ++j) {
            g[NX + j] += 2.0 * rweight(P, j) * u[j];
            cost += rweight(P, j) * u[j] * u[j];
        }
        const float* lam = S.lam + 3 + NLAM * k;
        for (int r = 0; r < NR; ++r) {
            double c, J[NL], sc;
            bool on, iq;
            brow<double, true>(r, P, St, (mi >> 10) & 1, (mi >> 11) & 1, x, u, dx, c, J, on, iq, sc);
            if (!on) continue;
            const double t = (double)lam[r] + beta * c;
            const double y = iq ? fmax(t, 0.0) : t;
            const double vr = iq ? fmax(c, 0.0) : fabs(c);
            viol = fmax(viol, vr / sc);
            if (!isfinite(c)) finite = false;
            for (int j = 0; j < NL; ++j) g[j] += y * J[j];
        }
        for (int j = 0; j < NWV; ++j) g64[NWV * k + j] = g[j];
        for (int i = 0; i < NX; ++i) g64b[NX * (k + 1) + i] = g[NWV + i];
    }
    __syncthreads();
    double stat = 0.0;
    for (int k = C.tid; k <= N; k += kBimThreads) {
        for (int i = 0; i < NX; ++i) {
            double gv = (k < N) ? g64[NWV * k + i] : 0.0;
            if (k > 0) gv += g64b[NX * k + i];
            if (k == N && i < 3) {
                const double e = (double)S.xh[i * Np1 + N] + (double)S.xl[i * Np1 + N] - P.goal[i];
                gv += 2.0 * P.wT * e;
                cost += P.wT * e * e;
            }
            if (k == 0 && i < 3) {
                const double c = (double)S.xh[i * Np1] + (double)S.xl[i * Np1] - P.start[i];
                gv += (double)S.lam[i] + beta * c;
                viol = fmax(viol, fabs(c));
            }
            stat = fmax(stat, fabs(gv));
            if (!isfinite(gv)) finite = false;
        }
        if (k < N)
            for (int j = 0; j < NU; ++j) stat = fmax(stat, fabs(g64[NWV * k + NX + j]));
    }
    // block reductions (double, through the workspace scratch)
    for (int o = 16; o > 0; o >>= 1) {
        cost += __shfl_xor_sync(kFullB, cost, o);
        viol = fmax(viol, __shfl_xor_sync(kFullB, viol, o));
        stat = fmax(stat, __shfl_xor_sync(kFullB, stat, o));
    }
    const bool fin = __all_sync(kFullB, finite);
    __syncthreads();
    double* red = g64b + NX * (N + 1);
    if (C.lane == 0) {
        red[C.warp] = cost;
        red[4 + C.warp] = viol;
        red[8 + C.warp] = stat;
        red[12 + C.warp] = fin ? 1.0 : 0.0;
    }
    __syncthreads();
    BCert ct;
    ct.cost = red[0] + red[1] + red[2] + red[3];
    ct.viol = fmax(fmax(red[4], red[5]), fmax(red[6], red[7]));
    ct.stat = fmax(fmax(red[8], red[9]), fmax(red[10], red[11]));
    ct.finite = red[12] > 0 && red[13] > 0 && red[14] > 0 && red[15] > 0 && isfinite(ct.cost);
    __syncthreads();
    return ct;
}

__global__ void __launch_bounds__(kBimThreads, 4) bimanual_kernel(EvalArgs A) {
    extern __shared__ float bsm[];
    BCtx C;
    C.tid = threadIdx.x;
    C.warp = threadIdx.x >> 5;
    C.lane = threadIdx.x & 31;
    C.S = bcarve(bsm, A.Nmax);
    C.rec = A.ws + (size_t)blockIdx.x * A.ws_per_warp;
    C.jac = C.rec + (size_t)kBimRec * A.Nmax;
    C.Nmax = A.Nmax;
    BSmem& S = C.S;
    // where lane i's entry of row r lies in a Jacobian record (its zero if the
    // row's pattern does not have the lane's variable)
    for (int t = C.tid; t < NR * 32; t += kBimThreads) {
        const int r = t >> 5, i = t & 31;
        int at = J_ZERO;
        for (int q = 0; q < 10 && bnz(r, q) >= 0; ++q)
            if (i < NL && bnz(r, q) == evar(i)) at = bnz_first(r) + q;
        S.at[t] = (uint16_t)(4 * at);
    }
    __syncthreads();
    const SolverParams& sp = A.sp;
    const int64_t n_tos = A.d_n ? min(*A.d_n, A.n) : A.n;
    __shared__ unsigned int s_t;
    for (;;) {
        if (C.tid == 0) s_t = atomicAdd(A.queue, 1u);
        __syncthreads();
        const unsigned int t = s_t;
        __syncthreads();
        if ((int64_t)t >= n_tos) break;
        const int64_t ti = A.perm ? (int64_t)A.perm[t] : (int64_t)t;
        const comet_mode_seq sq = A.seqs[ti];
        bool bad = sq.instance < 0 || sq.instance >= A.n_inst;
        const DevInstance* D = bad ? A.inst : A.inst + sq.instance;
        const int len = sq.len;
        bad = bad || len < 1 || len > D->Lmax || len > COMET_MAX_SEGMENTS;
        if (!bad)
            for (int i = 0; i < len; ++i) bad = bad || sq.modes[i] >= D->n_modes;
        if (bad) {
            if (C.tid == 0) {
                atomicExch(A.bad_input, 1);
                A.out_status[ti] = COMET_TO_NONFINITE;
                A.out_cost[ti] = __int_as_float(0x7fc00000);
                if (A.out_iters) A.out_iters[ti] = 0;
                if (A.out_viol) A.out_viol[ti] = __int_as_float(0x7fc00000);
                if (A.out_merit) A.out_merit[ti] = __int_as_float(0x7fc00000);
                if (A.out_stat) A.out_stat[ti] = __int_as_float(0x7fc00000);
            }
            continue;
        }
        C.D = D;
        load_inst(*D, C.P);
        C.len = len;
        C.N = D->K * len;
        C.Np1 = C.N + 1;
        const int N = C.N, Np1 = C.Np1, Nm1 = A.Nmax + 1;
        const BInst<float>& P = C.P;
        // initial iterate
        const float* warm = A.warm ? A.warm + ti * A.stride : nullptr;
        for (int q = C.tid; q < NX * Np1; q += kBimThreads) {
            const int i = q / Np1, k = q - i * Np1;
            float x;
            if (warm) {
                x = warm[i * Nm1 + k];
            } else if (i < 3) {
                const float al = (float)k / (float)N;
                x = (1.f - al) * P.start[i] + al * P.goal[i];
            } else {
                x = 0.f;
            }
            S.xh[q] = x;
            S.xl[q] = 0.f;
        }
        for (int q = C.tid; q < NU * N; q += kBimThreads) {
            const int j = q / N, k = q - j * N;
            S.us[q] = warm ? warm[NX * Nm1 + j * A.Nmax + k] : ((j == ULN - 5) ? P.mg : 0.f);
        }
        for (int q = C.tid; q < 3 + NLAM * N; q += kBimThreads) S.lam[q] = 0.f;
        for (int q = C.tid; q < NWV * N + NX; q += kBimThreads) S.dz[q] = S.gr[q] = 0.f;
        for (int k = C.tid; k < N; k += kBimThreads) {
            const int seg = (int)(((long long)k * len) / N);
            const int m = sq.modes[seg];
            int mL = 0, mR = 0;
            if (k + 1 < N) {
                const int m1 = sq.modes[(int)(((long long)(k + 1) * len) / N)];
                const int hL0 = (m / 13) % 13, hL1 = (m1 / 13) % 13, hR0 = m % 13, hR1 = m1 % 13;
                const int fL0 = hL0 ? (hL0 - 1) / 3 : -1, fL1 = hL1 ? (hL1 - 1) / 3 : -1;
                const int fR0 = hR0 ? (hR0 - 1) / 3 : -1, fR1 = hR1 ? (hR1 - 1) / 3 : -1;
                mL = fL0 != fL1;
                mR = fR0 != fR1;
            }
            S.mi[k] = m | (mL << 10) | (mR << 11);
        }
        __syncthreads();

        float beta = sp.beta0, rho = sp.rho0, eta = INFINITY;
        int inner = 0, it = 0, status = COMET_TO_MAX_ITER;
        bool nonfinite = false;
        for (it = 0; it < sp.max_iters; ++it) {
            // (assemble, sweep) trips through one call site of each phase
            // (one inlined copy in the hot loop): the measures and model at
            // the iterate, the dual update at beta_old after a solved
            // subproblem, and reassembly at rising damping after a failed
            // sweep.  Every decision is taken on CTA-wide reductions, so all
            // threads follow the same trips.
            enum { kMeasure, kUpdate, kRetry };
            int trip = kMeasure, retries = 0;
            bool fac = false, done = false;
            float beta_old = beta;
            for (;;) {
                // rows, gradient and measures; a retry keeps them (only the
                // damping changed)
                BMeasures m;
                if (trip != kRetry) m = bphase_a(C, beta, trip == kUpdate, beta_old);
                if (trip == kMeasure) {
                    if (!m.finite) {
                        status = COMET_TO_NONFINITE;
                        nonfinite = true;
                        done = true;
                        break;
                    }
                    // stop test (Sec. III-C): scaled rows within eps_primal,
                    // rows in physical units within half eps_feas, and
                    // stationarity relative to max(1, |J|)
                    const float eps_d = sp.eps_dual * fmaxf(1.f, beta / sp.beta_ref) * fmaxf(1.f, fabsf(m.cost));
                    if (m.viol <= sp.eps_primal && m.vphys <= 0.5f * (float)sp.eps_feas && m.stat <= eps_d &&
                        m.comp <= sp.eps_comp) {
                        status = COMET_TO_CONVERGED;
                        done = true;
                        break;
                    }
                    const float omega = fmaxf(eps_d, sp.omega_ratio * m.viol);
                    const bool solved = m.stat <= omega;
                    if (solved || inner >= sp.max_inner) {
                        beta_old = beta;
                        if (solved && m.viol > sp.eps_primal && m.viol > sp.eta_ratio * eta)
                            beta = fminf(sp.beta_max, beta * sp.beta_growth);
                        eta = m.viol;
                        inner = 0;
                        trip = kUpdate;
                        continue;
                    }
                }
                bphase_m(C, beta, rho);
                fac = bphase_b(C, beta, rho);
                if (fac || retries >= sp.max_retries) break;
                ++retries;
                rho = fminf(sp.rho_max, rho * 10.f);
                trip = kRetry;
            }
            if (done) break;
            ++inner;
            if (!fac) continue;
            bphase_gains(C);
            const float Dv = bphase_c(C);
            const float alpha = bphase_d(C, beta, Dv, sp);
            if (alpha > 0.f) {
                bphase_e(C, alpha);
                rho = fmaxf(sp.rho_min, rho / 10.f);
            } else {
                rho = fminf(sp.rho_max, rho * 10.f);
            }
        }
        const BCert ct = bcertify(C, beta);
        if (!ct.finite) nonfinite = true;
        if (nonfinite) status = COMET_TO_NONFINITE;
        if (status == COMET_TO_CONVERGED && !(ct.viol <= sp.eps_feas)) status = COMET_TO_INFEASIBLE;
        if (C.tid == 0) {
            A.out_status[ti] = status;
            A.out_cost[ti] = (float)ct.cost;
            if (A.out_viol) A.out_viol[ti] = (float)ct.viol;
            if (A.out_merit) A.out_merit[ti] = (float)(ct.cost + sp.merit_mu * fmax(ct.viol - sp.eps_feas, 0.0));
            if (A.out_iters) A.out_iters[ti] = it;
            if (A.out_stat) A.out_stat[ti] = (float)ct.stat;
        }
        if (A.out_traj) {
            float* out = A.out_traj + ti * A.stride;
            for (int q = C.tid; q < NX * Nm1; q += kBimThreads) {
                const int i = q / Nm1, k = q - i * Nm1;
                out[q] = (k <= N) ? S.xh[i * Np1 + k] + S.xl[i * Np1 + k] : 0.f;
            }
            for (int q = C.tid; q < NU * A.Nmax; q += kBimThreads) {
                const int j = q / A.Nmax, k = q - j * A.Nmax;
                out[NX * Nm1 + q] = (k < N) ? S.us[j * N + k] : 0.f;
            }
        }
        __syncthreads();
    }
}

}  // namespace

size_t bim_smem_bytes(int Nmax) { return bsmem_floats(Nmax) * sizeof(float); }

namespace {
SmemLimit g_smem_limit;
cudaError_t set_smem(size_t smem) {
    return cudaFuncSetAttribute(bimanual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
}  // namespace

int bim_blocks_per_sm(int Nmax) {
    const size_t smem = bim_smem_bytes(Nmax);
    if (g_smem_limit.raise(smem, set_smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, bimanual_kernel, kBimThreads, smem) != cudaSuccess)
        return 0;
    return nb;
}

cudaError_t launch_bimanual(const EvalArgs& a, int n_ctas, cudaStream_t s) {
    const size_t smem = bim_smem_bytes(a.Nmax);
    return launch_persistent(bimanual_kernel, n_ctas, kBimThreads, smem, s, a);
}

}  // namespace comet
