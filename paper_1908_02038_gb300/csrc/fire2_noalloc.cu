// Allocation-free energy/force evaluation (fire_energy_forces_noalloc).
//
// Some callers cannot call cudaMalloc at the point where they need forces:
// plug-ins of host programs whose memory pool owns all device memory and
// forbids stray allocations, and latency-critical loops where an allocation
// could synchronise the device or fail under memory pressure.  This entry
// point serves them: the caller passes device buffers for the
// positions and the results, and the only scratch the kernels need (per-atom
// energies and embedding derivatives) lives in the file-scope device array
// `g_scratch` below, sized for at most kNoAllocMaxAtoms atoms.  Every GPU that loads the library holds that array
// (about 0.5 MiB) until the process exits.
//
// The evaluation is all-pairs (minimum image), each atom summing over every
// other atom, so no neighbour list is needed and nothing accumulates across
// warps: every scratch value read in a call is written earlier in the same
// call.  One warp works on an atom (or four).  It tests 32 candidates at a time in FP32
// (FP64 issues at 1/58 of the FP32 rate on this part) against the cut-off plus
// the FP32 error of the coordinates, keeps those that pass in a short list in
// shared memory, and evaluates 32 list entries at a time in FP64, which
// decides the cut-off.  3,960 atoms: 141 us against 7,460 us with a thread
// per atom and every pair in FP64 (31 blocks on 152 SMs, 16 FP64 instructions
// for each of the 16 M pairs, twice); what remains is about half the FP64 pipe
// in the ~54 pairs per atom and half the FP32 tests.  Calls that overlap on the GPU (two streams, or two host threads) race
// on g_scratch and must be serialised by the caller.
#include <cuda.h>   // CUcontext and the driver function types (entry points, no link)
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>

#include "fire2.h"
#include "fire2_common.cuh"
#include "fire2_table.cuh"

void fire2_set_global_error(const char* msg);  // defined in fire2_api.cu (hidden)

namespace {

constexpr int kNoAllocMaxAtoms = 32768;
constexpr int kWarps = 8;              // warps per block
constexpr int kBlock = 32 * kWarps;    // candidates staged at a time, one per thread
// From here on a warp takes four atoms, which share the staging and the loads of
// the candidates (one / four atoms per warp: 3,999 atoms 141 / 174 us, with
// too few blocks; 10,975 atoms 1,241 / 851 us before the FP64 work was cut).
constexpr int kManyAtoms = 8192;
constexpr int kScratchDoubles = 2 * kNoAllocMaxAtoms;

// [0, N): energy of atom i; [N, 2N): F'(rho_i).
static __device__ __align__(256) double g_scratch[kScratchDoubles];

struct NaPot {
    int kind;
    double rc2;
    double eps, sigma2, lj_shift;
    double A, xi2, p, q2, r0inv, p_r0, q2_r0, rs, winv;
    double L[3], Linv[3];
    int per[3];
    fire2::ExpC ex;
    // FP32 candidate test
    float Lf[3], Linvf[3], rcf;
    float wrap[3];         // coordinates beyond this magnitude are wrapped first (periodic axes)
};

__device__ __noinline__ double na_image(double d, double L, double Linv) { return d - L * rint(d * Linv); }

// Minimum image of d, d - L rint(d / L); unchanged (no FP64 instruction) where
// |d| <= L / 2, by the bit patterns.
__device__ __forceinline__ void na_min_image(double& d, double L, double Linv, int per) {
    if (per && __double_as_longlong(fabs(d)) > __double_as_longlong(0.5 * L)) d = na_image(d, L, Linv);
}

__device__ __forceinline__ double na_warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 2^(j/256), the table of exp_tang, as products of 2^(k/16) and 2^(k/256).
__device__ __forceinline__ void na_exp_table(double* tab) {
    __shared__ double part[32];
    const int t = threadIdx.x;
    if (t < 32) part[t] = exp2(t < 16 ? t / 16.0 : (t - 16) / 256.0);
    __syncthreads();
    if (t < fire2::kExpTableSize) tab[t] = part[t >> 4] * part[16 + (t & 15)];
    __syncthreads();
}

// e^x in FP64; FAST: the exponents lie in exp_tang's range.
template <bool FAST>
__device__ __forceinline__ double na_exp(const NaPot& P, double x, const double* tab) {
    return FAST ? fire2::exp_tang(x, P.ex, tab) : exp(x);
}

// r and 1/r of a pair.  The exponentials multiply r's error by up to p r / r0, so
// r2 / sqrt(r2) gets its residual put back, which rounds it as sqrt does: forces
// of 3,960 Cu atoms off by 2.15e-15 as with the IEEE operations, 2.71e-15 without.
__device__ __forceinline__ void na_radius(double r2, double& r, double& rinv) {
    rinv = fire2::rsqrt_f64(r2);
    const double s = r2 * rinv;
    r = __double_as_longlong(r2) > 0 ? fma(fma(-s, s, r2), 0.5 * rinv, s) : 0.0;
}

// RGL pair terms: phi = A e^{-p s} S, g = xi^2 e^{-2q s} S, s = r/r0 - 1, with
// the quintic taper S on [rs, rc); returns the derivatives too.
template <bool FAST>
__device__ __forceinline__ void na_rgl_pair(const NaPot& P, double r, const double* tab, double& phi,
                                            double& dphi, double& g, double& dg) {
    const double s = r * P.r0inv - 1.0;
    const double ep = P.A * na_exp<FAST>(P, -P.p * s, tab);
    const double eq = P.xi2 * na_exp<FAST>(P, -P.q2 * s, tab);
    double S = 1.0, dS = 0.0;
    if (r > P.rs) {
        const double t = (r - P.rs) * P.winv;
        const double t2 = t * t, t3 = t2 * t;
        S = 1.0 - 10.0 * t3 + 15.0 * t3 * t - 6.0 * t3 * t2;
        dS = (-30.0 * t2 + 60.0 * t3 - 30.0 * t3 * t) * P.winv;
    }
    phi = ep * S;
    dphi = ep * (-P.p_r0 * S + dS);
    g = eq * S;
    dg = eq * (-P.q2_r0 * S + dS);
}

// Out of line, so that their FP64 instructions are issued only when needed.
__device__ __noinline__ float na_to_float(double x) { return (float)x; }
__device__ __noinline__ float na_wrapped(double x, double L, double Linv) {
    return (float)(x - L * floor(x * Linv));
}

// FP32 copy of coordinate a for the candidate test: the coordinate itself
// within a few box lengths (or on an open axis), wrapped into the box beyond.
// Truncated on the integer pipes (off by less than 2^-23 of its size) where
// the exponent is an FP32 one: a conversion takes the FP64 pipe, and every
// block makes three for each candidate.
__device__ __forceinline__ float na_coord(const NaPot& P, int a, double x) {
    const unsigned hi = (unsigned)__double2hiint(x), ahi = hi & 0x7fffffffu;
    float f = 0.f;
    if (ahi - (897u << 20) < (254u << 20))
        f = __uint_as_float((hi & 0x80000000u) | ((ahi - (896u << 20)) << 3) |
                            ((unsigned)__double2loint(x) >> 29));
    else if (ahi >= (897u << 20))   // beyond FP32, or not finite
        f = na_to_float(x);
    if (P.per[a] && !(fabsf(f) <= P.wrap[a])) return na_wrapped(x, P.L[a], P.Linv[a]);
    return f;
}

// Walks the atoms j != i inside (or within FP32 error of) the cut-off of the
// warp's A atoms i = i0 .. i0 + A - 1, 32 at a time: eval(a, j) runs on the
// lanes that hold an entry of atom i0 + a.  All threads of the block enter
// (i >= n: no atom).  list: A x 64 entries per warp.
template <int A, typename Eval>
__device__ __forceinline__ void na_walk(const double* __restrict__ pos, int n, const NaPot& P, int i0,
                                        float4* tile, int (*list)[64], Eval eval) {
    const int lane = threadIdx.x & 31;
    float xi[A][3], reach2[A];
    int cnt[A];   // entries in the atom's list, below 32 between candidates
#pragma unroll
    for (int u = 0; u < A; ++u) {
        float reach = P.rcf;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            xi[u][a] = i0 + u < n ? na_coord(P, a, pos[3 * (size_t)(i0 + u) + a]) : 0.f;
            // a pair inside rc has |x_j| <= |x_i| + rc on an open axis and
            // |x_j| <= wrap on a periodic one; each copy is off by 2^-23 of its
            // size, the difference and the shift by half as much
            reach += 0x1p-20f * (fabsf(xi[u][a]) + (P.per[a] ? P.wrap[a] : P.rcf));
        }
        reach2[u] = reach * reach * 1.00001f;
        cnt[u] = 0;
    }
    for (int base = 0; base < n; base += kBlock) {
        const int j0 = base + threadIdx.x;
        __syncthreads();
        if (j0 < n) {
            const double* p = pos + 3 * (size_t)j0;
            tile[threadIdx.x] = make_float4(na_coord(P, 0, p[0]), na_coord(P, 1, p[1]),
                                            na_coord(P, 2, p[2]), 0.f);
        }
        __syncthreads();
        const int m = min(kBlock, n - base);
        if (i0 >= n) continue;
        for (int k0 = 0; k0 < m; k0 += 32) {   // the warp stays together
            const int k = k0 + lane;
            const float4 x = tile[min(k, m - 1)];
            bool hit[A];
            bool any = false;
#pragma unroll
            for (int u = 0; u < A; ++u) {
                float d[3] = {x.x - xi[u][0], x.y - xi[u][1], x.z - xi[u][2]};
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    if (P.per[a]) {   // round to the nearest integer by 1.5 2^23 (|shift| <= 8)
                        const float r = __fadd_rn(__fmaf_rn(d[a], P.Linvf[a], 0x1.8p23f), -0x1.8p23f);
                        d[a] -= r * P.Lf[a];
                    }
                hit[u] = !(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] > reach2[u]) &&   // NaN: FP64
                         k < m && i0 + u < n && base + k != i0 + u;                  // decides
                any |= hit[u];
            }
            if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
            for (int u = 0; u < A; ++u) {
                const unsigned b = __ballot_sync(0xffffffffu, hit[u]);
                if (hit[u]) list[u][cnt[u] + __popc(b & ((1u << lane) - 1u))] = base + k;
                cnt[u] += __popc(b);
                if (cnt[u] >= 32) {
                    __syncwarp();
                    const int j = list[u][lane], rest = list[u][32 + lane];
                    eval(u, j);
                    __syncwarp();
                    list[u][lane] = rest;
                    cnt[u] -= 32;
                    __syncwarp();
                }
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < A; ++u)
        if (lane < cnt[u]) eval(u, list[u][lane]);
}

// Separation x_j - x_i (minimum image) in FP64; returns r^2.
__device__ __forceinline__ double na_sep(const double* __restrict__ pos, const NaPot& P,
                                         const double x[3], int j, double d[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        d[a] = pos[3 * (size_t)j + a] - x[a];
        na_min_image(d[a], P.L[a], P.Linv[a], P.per[a]);
    }
    return d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
}

// Pass 1 (RGL): F'(rho_i) and the per-atom energy, all-pairs.
// LJ: the whole evaluation (forces and energy) in this one pass.
template <int A, bool RGL, bool FAST>
__global__ void __launch_bounds__(kBlock) k_na_pass1(const double* __restrict__ pos, int n,
                                                     NaPot P, double* scratch,
                                                     double* __restrict__ forces) {
    __shared__ float4 tile[kBlock];
    __shared__ int list[kWarps][A][64];
    __shared__ double tab[fire2::kExpTableSize];
    if (RGL) na_exp_table(tab);
    const int w = threadIdx.x >> 5, i0 = (blockIdx.x * kWarps + w) * A;
    double x[A][3], s0[A], e[A], f[A][3];   // s0: density
#pragma unroll
    for (int u = 0; u < A; ++u) {
        s0[u] = e[u] = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[u][a] = 0.0;
            x[u][a] = i0 + u < n ? pos[3 * (size_t)(i0 + u) + a] : 0.0;
        }
    }
    na_walk<A>(pos, n, P, i0, tile, list[w], [&](int u, int j) {
        double d[3];
        const double r2 = na_sep(pos, P, x[u], j, d);
        if (!fire2::below_nonneg(r2, P.rc2)) return;
        if (RGL) {
            double r, rinv, phi, dphi, g, dg;
            na_radius(r2, r, rinv);
            na_rgl_pair<FAST>(P, r, tab, phi, dphi, g, dg);
            s0[u] += g;
            e[u] += phi;
        } else {
            const double ir2 = __drcp_rn(r2);
            const double sr2 = P.sigma2 * ir2;
            const double sr6 = sr2 * sr2 * sr2;
            e[u] += 0.5 * (4.0 * P.eps * (sr6 * sr6 - sr6) - P.lj_shift);
            const double q = 24.0 * P.eps * (2.0 * sr6 * sr6 - sr6) * ir2;
#pragma unroll
            for (int a = 0; a < 3; ++a) f[u][a] -= q * d[a];
        }
    });
#pragma unroll
    for (int u = 0; u < A; ++u) {
        if (i0 + u >= n) return;
        double en = na_warp_sum(e[u]);
        if (RGL) {
            double sq, fp;
            fire2::rgl_embed(na_warp_sum(s0[u]), sq, fp);
            en -= sq;
            if ((threadIdx.x & 31) == 0) scratch[kNoAllocMaxAtoms + i0 + u] = fp;
        } else if (forces) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double v = na_warp_sum(f[u][a]);
                if ((threadIdx.x & 31) == 0) forces[3 * (size_t)(i0 + u) + a] = v;
            }
        }
        if ((threadIdx.x & 31) == 0) scratch[i0 + u] = en;
    }
}

// Pass 2 (RGL): F_i = sum_j [2 phi'(r) + (F'_i + F'_j) g'(r)] (x_j - x_i) / r.
template <int A, bool FAST>
__global__ void __launch_bounds__(kBlock) k_na_pass2(const double* __restrict__ pos, int n,
                                                     NaPot P, const double* scratch,
                                                     double* __restrict__ forces) {
    __shared__ float4 tile[kBlock];
    __shared__ int list[kWarps][A][64];
    __shared__ double tab[fire2::kExpTableSize];
    na_exp_table(tab);
    const int w = threadIdx.x >> 5, i0 = (blockIdx.x * kWarps + w) * A;
    const double* fp = scratch + kNoAllocMaxAtoms;
    double x[A][3], fpi[A], f[A][3];
#pragma unroll
    for (int u = 0; u < A; ++u) {
        fpi[u] = i0 + u < n ? fp[i0 + u] : 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[u][a] = 0.0;
            x[u][a] = i0 + u < n ? pos[3 * (size_t)(i0 + u) + a] : 0.0;
        }
    }
    na_walk<A>(pos, n, P, i0, tile, list[w], [&](int u, int j) {
        double d[3];
        const double r2 = na_sep(pos, P, x[u], j, d);
        if (!fire2::below_nonneg(r2, P.rc2)) return;
        double r, rinv, phi, dphi, g, dg;
        na_radius(r2, r, rinv);
        na_rgl_pair<FAST>(P, r, tab, phi, dphi, g, dg);
        const double fs = (2.0 * dphi + (fpi[u] + fp[j]) * dg) * rinv;
#pragma unroll
        for (int a = 0; a < 3; ++a) f[u][a] += fs * d[a];
    });
    if (!forces) return;
#pragma unroll
    for (int u = 0; u < A; ++u) {
        if (i0 + u >= n) return;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double v = na_warp_sum(f[u][a]);
            if ((threadIdx.x & 31) == 0) forces[3 * (size_t)(i0 + u) + a] = v;
        }
    }
}

// Fixed-order sum of the atoms' energies into *energy (one block of 1024).
__global__ void __launch_bounds__(1024) k_na_energy(const double* scratch, int n, double* energy) {
    __shared__ double sh[32];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) s += scratch[k];
    s = na_warp_sum(s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    s = na_warp_sum(sh[threadIdx.x]);
    if (threadIdx.x == 0 && energy) *energy = s;
}

std::mutex g_mu;

// The scratch array's device address is looked up once per device context:
// cudaDeviceReset (or a reset of the primary context) gives the device a new
// context and reloads the module, so the cache is keyed on the context's
// unique id (cuCtxGetId, through the runtime's driver entry points).
struct ScratchAddr {
    unsigned long long ctx_id = 0;   // 0 = none cached
    double* ptr = nullptr;
};
ScratchAddr g_addr[128];

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

// Unique id of the current context, or 0 when it cannot be had (then the
// address is looked up on every call).
unsigned long long current_context_id() {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static bool resolved = false;
    if (!resolved) {   // under g_mu
        cudaDriverEntryPointQueryResult q1, q2;
        void* f1 = nullptr;
        void* f2 = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault,
                                             &q1) == cudaSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault,
                                             &q2) == cudaSuccess &&
            q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
            get_current = reinterpret_cast<CtxGetCurrentFn>(f1);
            get_id = reinterpret_cast<CtxGetIdFn>(f2);
        }
        resolved = true;
    }
    if (!get_current || !get_id) return 0;
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (get_current(&c) != CUDA_SUCCESS || !c || get_id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of g_scratch in the current device's context.
cudaError_t scratch_address(double** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    const unsigned long long id = current_context_id();
    ScratchAddr& a = g_addr[dev];
    if (id == 0 || a.ctx_id != id || !a.ptr) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);   // also makes the context current
        if (e != cudaSuccess) return e;
        a.ptr = static_cast<double*>(p);
        a.ctx_id = current_context_id();
    }
    *out = a.ptr;
    return cudaSuccess;
}

fire_status na_fail(fire_status code, const char* msg) {
    fire2_set_global_error(msg);
    return code;
}

}  // namespace

extern "C" fire_status fire_energy_forces_noalloc(const fire_potential_t* pot, int64_t n_atoms,
                                                  const int32_t periodic[3], const double* d_pos,
                                                  const double box[3], double* d_forces,
                                                  double* d_energy, void* stream) {
    if (!pot || !periodic || !d_pos || !box)
        return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: NULL argument");
    if (n_atoms < 1 || n_atoms > kNoAllocMaxAtoms) {
        char buf[160];
        snprintf(buf, sizeof buf,
                 "fire_energy_forces_noalloc: n_atoms = %lld outside [1, %d] (size of the "
                 "static scratch array)", (long long)n_atoms, kNoAllocMaxAtoms);
        return na_fail(FIRE_ERR_ARG, buf);
    }
    if (pot->precision != FIRE_PREC_FP64)
        return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: only FIRE_PREC_FP64");
    NaPot P{};
    P.kind = pot->kind;
    double rc = 0.0;
    bool fast = true;   // the exponents lie in exp_tang's range (|x| < 700)
    if (pot->kind == FIRE_POT_LJ) {
        if (!(pot->rc_lj > 0.0 && pot->sigma > 0.0 && pot->eps > 0.0))
            return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: LJ needs eps, sigma, rc_lj > 0");
        rc = pot->rc_lj;
        P.eps = pot->eps;
        P.sigma2 = pot->sigma * pot->sigma;
        const double sr6 = std::pow(pot->sigma / pot->rc_lj, 6.0);
        P.lj_shift = 4.0 * pot->eps * (sr6 * sr6 - sr6);
    } else if (pot->kind == FIRE_POT_RGL) {
        if (!(pot->rc > pot->rs && pot->rs > 0.0 && pot->r0 > 0.0 && pot->xi > 0.0 && pot->A >= 0.0))
            return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: bad RGL parameters");
        rc = pot->rc;
        P.A = pot->A;
        P.xi2 = pot->xi * pot->xi;
        P.p = pot->p;
        P.q2 = 2.0 * pot->q;
        P.r0inv = 1.0 / pot->r0;
        P.p_r0 = pot->p / pot->r0;
        P.q2_r0 = 2.0 * pot->q / pot->r0;
        P.rs = pot->rs;
        P.winv = 1.0 / (pot->rc - pot->rs);
        double table[fire2::kExpTableSize];
        P.ex = fire2::make_exp_constants(table);
        const double smax = std::fmax(1.0, rc / pot->r0 - 1.0);
        fast = std::fabs(P.p) * smax < 600.0 && std::fabs(P.q2) * smax < 600.0;
    } else {
        return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: unknown potential kind");
    }
    P.rc2 = rc * rc;
    P.rcf = (float)rc;
    for (int a = 0; a < 3; ++a) {
        if (!(box[a] > 0.0) || !std::isfinite(box[a]))
            return na_fail(FIRE_ERR_ARG, "fire_energy_forces_noalloc: box lengths must be > 0");
        if (periodic[a] && box[a] < 2.0 * rc)
            return na_fail(FIRE_ERR_ARG,
                           "fire_energy_forces_noalloc: periodic box shorter than twice the cut-off");
        P.L[a] = box[a];
        P.Linv[a] = 1.0 / box[a];
        P.per[a] = periodic[a] ? 1 : 0;
        P.Lf[a] = (float)box[a];
        P.Linvf[a] = (float)P.Linv[a];
        P.wrap[a] = 4.f * P.Lf[a];
    }
    double* scratch = nullptr;
    cudaError_t e = scratch_address(&scratch);
    if (e != cudaSuccess) return na_fail(FIRE_ERR_CUDA, cudaGetErrorString(e));
    int n = (int)n_atoms;
    const int A = n >= kManyAtoms && fast ? 4 : 1, blocks = (n + kWarps * A - 1) / (kWarps * A);
    cudaStream_t s = (cudaStream_t)stream;
    // cudaLaunchKernel returns the status of its own launch, so an error left
    // pending by the caller's earlier work is neither reported as this call's
    // nor cleared
    const double* pos = d_pos;
    double* fout = d_forces;
    double* eout = d_energy;
    void* args12[] = {(void*)&pos, (void*)&n, (void*)&P, (void*)&scratch, (void*)&fout};
    const bool rgl = P.kind == FIRE_POT_RGL;
    const void *pass1, *pass2 = nullptr;
    if (!rgl)
        pass1 = A == 4 ? (const void*)k_na_pass1<4, false, true> : (const void*)k_na_pass1<1, false, true>;
    else if (!fast)
        pass1 = (const void*)k_na_pass1<1, true, false>, pass2 = (const void*)k_na_pass2<1, false>;
    else if (A == 4)
        pass1 = (const void*)k_na_pass1<4, true, true>, pass2 = (const void*)k_na_pass2<4, true>;
    else
        pass1 = (const void*)k_na_pass1<1, true, true>, pass2 = (const void*)k_na_pass2<1, true>;
    e = cudaLaunchKernel(pass1, dim3(blocks), dim3(kBlock), args12, 0, s);
    if (e == cudaSuccess && rgl) e = cudaLaunchKernel(pass2, dim3(blocks), dim3(kBlock), args12, 0, s);
    void* args3[] = {(void*)&scratch, (void*)&n, (void*)&eout};
    if (e == cudaSuccess)
        e = cudaLaunchKernel((const void*)k_na_energy, dim3(1), dim3(1024), args3, 0, s);
    if (e != cudaSuccess) return na_fail(FIRE_ERR_CUDA, cudaGetErrorString(e));
    return FIRE_OK;
}
