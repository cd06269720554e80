// The relaxation loop of small and mid-size systems in one resident kernel.
//
// On a few thousand atoms an iteration of the kernel chain (fire2_device.cuh)
// is latency: five or six launches, each with its own loads of the state, its
// own reduction trees and its tail.  Here one cooperative launch (a block per
// SM, each owning a contiguous share of the atoms) runs iterations until the
// relaxation stops or the lists must be rebuilt; the graph's WHILE body is the
// list build followed by this kernel.  Positions, velocities and forces stay
// in the owner's shared memory; what others read goes through L2 (fixed-point
// records with F'(rho) for RGL, FP64 positions for LJ).  Per iteration:
//   RGL  densities and F' of the own atoms (full list)       | barrier
//        forces of the own atoms (full list, no atomics), the six reductions
//        of (F, v) as one row of partials per block          | barrier
//        every block adds up the rows in the same order, runs Algorithm 2 on
//        identical numbers and updates its atoms              | barrier
//   LJ   the same without the density pass.
// The full list costs each pair twice but needs no atomics, no clearing and no
// embedding pass, and an atom's sums end in its own threads, next to its
// velocity.  L lanes share an atom (group sums in FP64).
//
// A barrier is one atomic and a poll per block.  The launch is cooperative, so
// every block is resident; each wait ends after LoopC::wait_ns all the same, with
// an abort flag that every other wait and every later launch of the call sees.
// A block that finds its count complete goes on, whatever others have done by
// then, so it is the host that looks at the flag after the last launch: the call
// returns FIRE_ERR_TIMEOUT.
//
// One evaluation (LoopC::eval) is the same passes and sums, then the export: 497
// atoms 130 -> 102 us a call, list build and copies included.
//
// us per iteration, chain / resident loop (152 SMs): LJ 255 atoms 21.8 / 12.4,
// 2,915 atoms 45 / 23, 10,975 atoms 80 / 53; RGL 255 atoms 30 / 14.3, 3,999 atoms
// 40.5 / 18.9, 10,975 atoms 46 / 29, 31,999 atoms 69 / 41.0, 62,499 atoms 98 / 77.
// A barrier takes 1.3 us, the control step about 2, the sums of the rows 0.8; the
// rest is the pair passes, which from ~10,000 atoms are bound by issue.
#pragma once

#include "fire2_device.cuh"

namespace fire2 {

constexpr int kLoopThreads = 1024;
constexpr int kLoopRows = 7;   // P, |F|^2, |v|^2, E, max |F_i|^2, max |F_i,d|, status
constexpr unsigned long long kLoopWaitNs = 5000000000ull;
constexpr unsigned kLoopSpan = 1u << 31;   // half of what the low half holds

struct LoopC {
    double* rows;          // kLoopRows x gridDim.x partials
    int share;             // atoms per block (the last block may have fewer)
    int eval;              // 1: one evaluation (F to b.f and b.f_out, E to b.e_out)
    unsigned long long wait_ns;   // limit of a wait; 0: every wait runs out (tests)
    unsigned span;         // arrivals after which the blocks leave for a list, due or not
};

// Shared-memory bytes of a block that owns `share` atoms.
inline size_t loop_smem(int share) { return (size_t)share * (9 * sizeof(double) + 3 * sizeof(float)); }

struct LoopShared {
    FireParamsD prm;
    FireScal fs;
    double sum[kLoopRows];
    double red[6][32];
    int ok, votes, stop, status;
};

// All blocks' writes before the barrier are visible after it (to loads that
// bypass L1).  The counter's low half counts arrivals since the last list build,
// its high half the votes that came with them; votes receives whether there was
// any.  The arrivals must not carry into the votes, which some blocks would see
// and others not: the blocks leave for a list (which resets the counter) beyond
// LoopC::span.  False once any wait of the grid has run out.
__device__ __forceinline__ bool loop_barrier(DevState* st, unsigned& target, LoopShared& sh,
                                             unsigned long long wait_ns, bool vote, bool& votes) {
    target += gridDim.x;
    const int mine = __syncthreads_or(vote);
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;"
                     :: "l"(&st->bar), "l"(1ull + (mine ? 1ull << 32 : 0ull)) : "memory");
        const unsigned goal = target + (wait_ns == 0ull ? 1u : 0u);   // one more never comes
        unsigned long long t0 = 0ull, v;
        int ok = 1;
        for (int n = 0;; ++n) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&st->bar) : "memory");
            if ((int)((unsigned)v - goal) >= 0) break;
            if ((n & 255) != 255) continue;
            const unsigned long long t = globaltimer_ns();
            if (t0 == 0ull) t0 = t;
            if (*(volatile unsigned*)&st->bar_abort != 0u || t - t0 >= wait_ns) {
                atomicExch(&st->bar_abort, 1u);
                ok = 0;
                break;
            }
        }
        sh.ok = ok;
        sh.votes = (v >> 32) != 0ull;
    }
    __syncthreads();
    votes = sh.votes != 0;
    return sh.ok != 0;
}

__device__ __forceinline__ lvec4 ld_lvec4_l2(const lvec4* p) {
    const longlong2* q = reinterpret_cast<const longlong2*>(p);
    const longlong2 a = __ldcg(q), b = __ldcg(q + 1);
    return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void ld_pos_l2(const dvec4* p, double& x, double& y, double& z) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p));
    x = a.x;
    y = a.y;
    z = __ldcg(reinterpret_cast<const double*>(p) + 2);
}

// Density pass over the block's atoms: F'(rho) into the atoms' records; returns
// this thread's energy.
template <int L>
__device__ __forceinline__ double loop_density(const Bufs& b, const PotC& P, const long long* qt,
                                               int i0, int own) {
    const int lane = threadIdx.x % L;
    double e = 0.0;
    for (int a = threadIdx.x / L; a < own; a += blockDim.x / L) {
        const int i = i0 + a, m = b.nnbr[i];
        const lvec4 qi = ld_lvec4_l2(b.xq64 + i);
        ffloat2 acc = {{0.f, 0.f}, {0.f, 0.f}};   // repulsive energy, density
        // the atom one pair ahead and the entry two ahead load meanwhile
        uint32_t e_nx = lane < m ? b.nbr[(size_t)lane * b.n + i] : (uint32_t)i;
        uint32_t e_n2 = lane + L < m ? b.nbr[(size_t)(lane + L) * b.n + i] : (uint32_t)i;
        lvec4 q_nx = ld_lvec4_l2(b.xq64 + (e_nx & kIdxMask));
        for (int k = lane; k < m; k += L) {
            const uint32_t en = e_nx;
            const lvec4 qj = q_nx;
            e_nx = e_n2;
            if (k + L < m) q_nx = ld_lvec4_l2(b.xq64 + (e_nx & kIdxMask));
            if (k + 2 * L < m) e_n2 = b.nbr[(size_t)(k + 2 * L) * b.n + i];
            const ffloat r2 = ff_norm2(pair_sep_ff(qt, qi, qj, en));
            const bool rows = ff_in_rows(P.ff, r2.hi);
            if (!rows && !(r2.hi < P.ff.rc2)) continue;
            ffloat2 v;
            if (rows) {
                v = ff_eval2(b.tab_ffd, P.ff, r2);
            } else {
                double rinv, phi, dphi, gg, dg;
                rgl_pair64(P, P.lam2 * ff_to_f64(r2), b.exp_table, rinv, phi, dphi, gg, dg);
                const ffloat p = f64_to_ff(phi), q = f64_to_ff(gg);
                v = {make_float2(p.hi, q.hi), make_float2(p.lo, q.lo)};
            }
            acc = ff_acc2(acc, v);
        }
        // lane 0: the repulsive energy; lane L / 2: the density
        const double s = group_sum2<L>(ff_to_f64(ff_first(acc)), ff_to_f64(ff_second(acc)));
        if (lane == 0) e += s;
        if (lane == L / 2) {
            double sq, fp;
            ffloat fpf;
            rgl_embed_dd(s, sq, fp, fpf);
            fp_store(b, i, fpf);
            e -= sq;
        }
    }
    return e;
}

// Component lane / (L / 4) of atom a's force (group_sum4) into f, 0 where frozen.
template <int L>
__device__ __forceinline__ void loop_store(const Bufs& b, int i, int a, int lane, int share, double s,
                                           double* f) {
    const int q = lane / (L / 4);
    if (lane % (L / 4) != 0 || q == 3) return;
    const unsigned m = b.dofmask ? b.dofmask[i] : 0u;
    f[q * share + a] = (m >> q) & 1u ? 0.0 : s;
}

// Force pass over the block's atoms into f (three arrays of `share`).
template <int L>
__device__ __forceinline__ void loop_force(const Bufs& b, const PotC& P, const long long* qt, int i0,
                                           int own, int share, double* f) {
    const int lane = threadIdx.x % L;
    for (int a = threadIdx.x / L; a < own; a += blockDim.x / L) {
        const int i = i0 + a, m = b.nnbr[i];
        const lvec4 qi = ld_lvec4_l2(b.xq64 + i);
        const ffloat fpi = fp_load(qi);
        ffloat2 fxy = {{0.f, 0.f}, {0.f, 0.f}};
        ffloat fz = {0.f, 0.f};
        uint32_t e_nx = lane < m ? b.nbr[(size_t)lane * b.n + i] : (uint32_t)i;
        uint32_t e_n2 = lane + L < m ? b.nbr[(size_t)(lane + L) * b.n + i] : (uint32_t)i;
        lvec4 q_nx = ld_lvec4_l2(b.xq64 + (e_nx & kIdxMask));
        for (int k = lane; k < m; k += L) {
            const uint32_t en = e_nx;
            const lvec4 qj = q_nx;
            e_nx = e_n2;
            if (k + L < m) q_nx = ld_lvec4_l2(b.xq64 + (e_nx & kIdxMask));
            if (k + 2 * L < m) e_n2 = b.nbr[(size_t)(k + 2 * L) * b.n + i];
            const ffvec d = pair_sep_ff(qt, qi, qj, en);
            const ffloat r2 = ff_norm2(d);
            const bool rows = ff_in_rows(P.ff, r2.hi);
            if (!rows && !(r2.hi < P.ff.rc2)) continue;
            ffloat c0, c1;
            if (rows) {
                const ffloat2 c = ff_eval2(b.tab_fff, P.ff, r2);
                c0 = ff_first(c);
                c1 = ff_second(c);
            } else {
                double rinv, phi, dphi, gg, dg;
                rgl_pair64(P, P.lam2 * ff_to_f64(r2), b.exp_table, rinv, phi, dphi, gg, dg);
                c0 = f64_to_ff(2.0 * dphi * rinv * P.lam);
                c1 = f64_to_ff(dg * rinv * P.lam);
            }
            const ffloat fs = ff_madd(ff_add(fpi, fp_load(qj)), c1, c0);
            const ffloat2 t = ff_mul2_neg(fs, d.xy);
            fxy = ff_acc2_neg(fxy, t.hi, t.lo);
            fz = ff_acc(fz, ff_mul_nn(fs, d.z));
        }
        const double s = group_sum4<L>(ff_to_f64(ff_first(fxy)), ff_to_f64(ff_second(fxy)),
                                       ff_to_f64(fz), 0.0);
        loop_store<L>(b, i, a, lane, share, s, f);
    }
}

// Lennard-Jones forces and energy, each pair from both ends.
template <int L>
__device__ __forceinline__ double loop_force_lj(const Bufs& b, const PotC& P, const double3* tbl, int i0,
                                                int own, int share, const double* x, double* f) {
    const int lane = threadIdx.x % L;
    double et = 0.0;
    for (int a = threadIdx.x / L; a < own; a += blockDim.x / L) {
        const int i = i0 + a, m = b.nnbr[i];
        const double xi = x[a], yi = x[share + a], zi = x[2 * share + a];
        double fx = 0.0, fy = 0.0, fz = 0.0, ep = 0.0;
        for (int k = lane; k < m; k += L) {
            const uint32_t e = b.nbr[(size_t)k * b.n + i];
            const int code = (int)(e >> kIdxBits);
            double dx, dy, dz;
            ld_pos_l2(b.x + (e & kIdxMask), dx, dy, dz);
            dx -= xi;
            dy -= yi;
            dz -= zi;
            if (code != kCodeZero) {
                const double3 s = tbl[code];
                dx -= s.x;
                dy -= s.y;
                dz -= s.z;
            }
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (!below_nonneg(r2, P.rc2)) continue;
            const double ir2 = rcp_f64(r2);
            const double sr2 = P.sigma2 * ir2;
            const double sr6 = sr2 * sr2 * sr2;
            const double c = fma(sr6, sr6, -sr6);                       // sr12 - sr6
            ep += fma(4.0 * P.eps, c, -P.lj_shift);
            const double w = 24.0 * P.eps * fma(sr6, sr6, c) * ir2;
            fx = fma(-w, dx, fx);
            fy = fma(-w, dy, fy);
            fz = fma(-w, dz, fz);
        }
        const double s = group_sum4<L>(fx, fy, fz, ep);
        loop_store<L>(b, i, a, lane, share, s, f);
        if (lane == 3 * (L / 4)) et = fma(0.5, s, et);
    }
    return et;
}

// This block's row of partials: the six reductions of its (F, v), energy and
// status.
__device__ __forceinline__ void loop_partials(const RedAcc& a, int status, const LoopC& c, LoopShared& sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double s = warp_sum4(a.P, a.F2, a.V2, a.E);
    double m0 = warp_max_nonneg(a.fa2), m1 = warp_max_nonneg(a.fin);
    if ((lane & 7) == 0) sh.red[lane >> 3][w] = s;
    if (lane == 0) {
        sh.red[4][w] = m0;
        sh.red[5][w] = m1;
    }
    __syncthreads();
    if (w == 0) {
        const bool in = lane < nw;
        s = warp_sum4(in ? sh.red[0][lane] : 0.0, in ? sh.red[1][lane] : 0.0,
                      in ? sh.red[2][lane] : 0.0, in ? sh.red[3][lane] : 0.0);
        m0 = warp_max_nonneg(in ? sh.red[4][lane] : 0.0);
        m1 = warp_max_nonneg(in ? sh.red[5][lane] : 0.0);
        double* row = c.rows + blockIdx.x;
        const int G = gridDim.x;
        if ((lane & 7) == 0) row[(lane >> 3) * G] = s;
        if (lane == 0) {
            row[4 * G] = m0;
            row[5 * G] = m1;
            row[6 * G] = (double)status;
        }
    }
}

// All rows added up, the same in every block: warp r takes quantity r.
__device__ __forceinline__ void loop_sums(const LoopC& c, LoopShared& sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, G = gridDim.x;
    if (w < kLoopRows) {
        const double* row = c.rows + (size_t)w * G;
        double v = 0.0;
        if (w < 4) {
            for (int k = lane; k < G; k += 32) v += __ldcg(row + k);
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        } else {
            for (int k = lane; k < G; k += 32) v = max_nonneg(v, __ldcg(row + k));
            v = warp_max_nonneg(v);
        }
        if (lane == 0) sh.sum[w] = v;
    }
    __syncthreads();
}

// Algorithm 2 on the sums (thread 0 of every block, on the same numbers).
static __device__ __noinline__ void loop_control(LoopShared& sh) {
    const double *s = sh.sum, E = s[3];
    FireScal fs = sh.fs;
    bool stop = true;
    sh.status = (int)s[6];
    if (sh.status != ST_OK) {
        fs.evals += 1;
    } else if (!isfinite(E) || !isfinite(s[1]) || !isfinite(s[2])) {
        fs.evals += 1;
        sh.status = ST_NONFINITE;
    } else {
        stop = fire_control_step(sh.prm, fs, s[0], s[1], s[2], s[4], s[5]);
    }
    sh.fs = fs;
    sh.stop = stop ? 1 : 0;
}

// The end of one evaluation: forces, energy and state out.
__device__ __forceinline__ void loop_export(const Bufs& b, int i0, int own, int share, const double* f,
                                            const LoopShared& sh) {
    for (int a = threadIdx.x; a < own; a += blockDim.x)
        f_store(b, i0 + a, f[a], f[share + a], f[2 * share + a]);
    if (b.f_out)
        for (int k = threadIdx.x; k < 3 * own; k += blockDim.x)
            b.f_out[3 * (size_t)i0 + k] = f[(k % 3) * share + k / 3];
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    const double E = sh.sum[3], F2 = sh.sum[1];
    if (b.e_out) *b.e_out = E;
    b.st->energy = E;
    b.st->F2 = F2;
    b.st->fmax2 = sh.sum[4];
    b.st->finf = sh.sum[5];
    if (b.st->status == ST_OK && (!isfinite(E) || !isfinite(F2))) b.st->status = ST_NONFINITE;
}

// The element-wise step of the block's atoms; returns this thread's largest
// squared displacement since the list build.
template <bool RGL, bool KICK>
__device__ __forceinline__ float loop_update(const Bufs& b, const FireScal& s, int i0, int own, int share,
                                             double* x, double* v, const double* f, const float* xr) {
    float d2 = 0.f;
    for (int a = threadIdx.x; a < own; a += blockDim.x) {
        dvec4 xa = make_dvec4(x[a], x[share + a], x[2 * share + a], 0.0);
        dvec4 va = make_dvec4(v[a], v[share + a], v[2 * share + a], 0.0);
        const dvec4 fa = make_dvec4(f[a], f[share + a], f[2 * share + a], 0.0);
        fire_update_pre(s, xa, va, fa);
        fire_update_drift_k<KICK>(s, s.dt_cur, xa, va, fa);
        x[a] = xa.x;
        x[share + a] = xa.y;
        x[2 * share + a] = xa.z;
        v[a] = va.x;
        v[share + a] = va.y;
        v[2 * share + a] = va.z;
        if (RGL)
            b.xq64[i0 + a] = {to_fixed64(xa.x, b.fbits), to_fixed64(xa.y, b.fbits),
                              to_fixed64(xa.z, b.fbits), 0ll};
        else
            b.x[i0 + a] = xa;
        const float dx = f64_to_f32_trunc(xa.x) - xr[a], dy = f64_to_f32_trunc(xa.y) - xr[share + a],
                    dz = f64_to_f32_trunc(xa.z) - xr[2 * share + a];
        d2 = fmaxf(d2, dx * dx + dy * dy + dz * dz);
    }
    return d2;
}

template <bool RGL, int L, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_loop(Bufs b, PotC P, GeoC g, LoopC c,
                                                          cudaGraphConditionalHandle hw) {
    extern __shared__ double dyn[];
    __shared__ LoopShared sh;
    __shared__ long long qt[RGL ? 375 : 1];
    __shared__ double3 tbl[RGL ? 1 : 125];
    const int share = c.share, i0 = blockIdx.x * share, own = max(0, min(share, b.n - i0));
    double *x = dyn, *v = x + 3 * share, *f = v + 3 * share;
    float* xr = reinterpret_cast<float*>(f + 3 * share);
    DevState* st = b.st;
    if (threadIdx.x == 0) {
        sh.prm = st->prm;
        sh.fs = st->fs;
        sh.stop = 0;
        sh.status = st->status;
        sh.ok = st->bar_abort == 0u ? 1 : 0;
    }
    if (RGL)
        fill_qshift64_table(qt, g);
    else
        fill_shift_table(tbl, g);
    for (int a = threadIdx.x; a < own; a += blockDim.x) {
        const dvec4 xa = b.x[i0 + a], va = b.v[i0 + a];
        const float4 r = b.xf[i0 + a];
        x[a] = xa.x;
        x[share + a] = xa.y;
        x[2 * share + a] = xa.z;
        v[a] = va.x;
        v[share + a] = va.y;
        v[2 * share + a] = va.z;
        xr[a] = r.x;
        xr[share + a] = r.y;
        xr[2 * share + a] = r.z;
    }
    const unsigned long long budget = st->budget_ns, t_start = st->t_start;
    const float skin2 = (float)g.half_skin2;
    __syncthreads();
    const int status0 = sh.status;   // of the list build, the same for every block
    unsigned target = 0u;
    bool ok = sh.ok != 0, rebuild = false, votes;
    while (ok) {
        RedAcc acc;
        if (RGL) {
            acc.E = loop_density<L>(b, P, qt, i0, own);
            if (!(ok = loop_barrier(st, target, sh, c.wait_ns, false, votes))) break;
            loop_force<L>(b, P, qt, i0, own, share, f);
        } else {
            acc.E = loop_force_lj<L>(b, P, tbl, i0, own, share, x, f);
        }
        __syncthreads();
        const double vvh = sh.fs.vv ? sh.fs.vv_half : 0.0;
        for (int a = threadIdx.x; a < own; a += blockDim.x) {
            dvec4 va = make_dvec4(v[a], v[share + a], v[2 * share + a], 0.0);
            const dvec4 fa = make_dvec4(f[a], f[share + a], f[2 * share + a], 0.0);
            if (sh.fs.vv) {   // second half kick of velocity Verlet, with the new force
                va.x += vvh * fa.x;
                va.y += vvh * fa.y;
                va.z += vvh * fa.z;
                v[a] = va.x;
                v[share + a] = va.y;
                v[2 * share + a] = va.z;
            }
            acc.P = fma(fa.z, va.z, fma(fa.y, va.y, fma(fa.x, va.x, acc.P)));
            const double q = fma(fa.z, fa.z, fma(fa.y, fa.y, fa.x * fa.x));
            acc.F2 += q;
            acc.V2 = fma(va.z, va.z, fma(va.y, va.y, fma(va.x, va.x, acc.V2)));
            acc.fa2 = max_nonneg(acc.fa2, q);
            acc.fin = max_nonneg(acc.fin, max_nonneg(abs_bits(fa.x),
                                                     max_nonneg(abs_bits(fa.y), abs_bits(fa.z))));
        }
        int status = status0;
        if (blockIdx.x == 0 && budget && globaltimer_ns() - t_start > budget && status == ST_OK)
            status = ST_TIMEOUT;
        loop_partials(acc, status, c, sh);
        if (!(ok = loop_barrier(st, target, sh, c.wait_ns, false, votes))) break;
        loop_sums(c, sh);
        if (c.eval) {
            loop_export(b, i0, own, share, f, sh);
            return;
        }
        if (threadIdx.x == 0) loop_control(sh);
        __syncthreads();
        if (sh.stop) break;
        const float d2 = sh.fs.kick_after != 0.0
                             ? loop_update<RGL, true>(b, sh.fs, i0, own, share, x, v, f, xr)
                             : loop_update<RGL, false>(b, sh.fs, i0, own, share, x, v, f, xr);
        // an atom further than skin / 2 from where the lists were built, or the
        // barrier's count used up (the same in every block): all leave for a new list
        if (!(ok = loop_barrier(st, target, sh, c.wait_ns, d2 > skin2 || target > c.span, votes))) break;
        if (votes) {
            rebuild = true;
            break;
        }
    }
    if (c.eval) return;   // a wait has run out
    // positions and velocities back (the list build reads x; the next launch
    // both), the state by block 0
    for (int a = threadIdx.x; a < own; a += blockDim.x) {
        b.x[i0 + a] = make_dvec4(x[a], x[share + a], x[2 * share + a], 0.0);
        b.v[i0 + a] = make_dvec4(v[a], v[share + a], v[2 * share + a], 0.0);
    }
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    if (ok) {
        st->fs = sh.fs;
        st->P = sh.sum[0];
        st->F2 = sh.sum[1];
        st->V2 = sh.sum[2];
        st->energy = sh.sum[3];
        st->fmax2 = sh.sum[4];
        st->finf = sh.sum[5];
        if (sh.status != ST_OK) st->status = sh.status;
    }
    st->done = rebuild ? 0 : 1;
    cudaGraphSetConditional(hw, rebuild ? 1u : 0u);
}

}  // namespace fire2
