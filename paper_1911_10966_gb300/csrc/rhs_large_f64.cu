// Float64 residual at p = 15 (N = 16 LGL nodes per direction, 4096 nodes per element): the degree
// of the paper's cost comparison above the one-CTA-per-element range of rhs_fix.cuh (an element's
// float64 state, primitives and geometry no longer fit one SM's shared memory).  Same discretisation
// (eq. discEL, eq. MacroForm, eq. NSL), built in four passes over the element grid:
//   1. lg_volume_fix (ES-C, SF-KG; lg_volume for DC), one CTA per (element, direction l, plane of N lines
//      of direction l): the N(N-1)/2 distinct pairs of each line are evaluated once each, the two line ends
//      add the interface SAT of the faces normal to l; each direction writes its own residual part r_l
//      (scaled by 1/w_i) and, for mu > 0, theta_l = D_l w + lift of the entropy variables w.
//   2. lg_viscous (mu > 0), one thread per node: the physical gradient, tau and the heat flux, and the
//      contravariant viscous fluxes Ftilde_l, written over theta with their face traces.
//   3. lg_visc_div (mu > 0), one CTA per (element, l, plane): r_l += D_l Ftilde_l along the lines
//      plus the BR1 interface term (E_ii/2)(Ftilde_nbr - Ftilde_own)/w_i at the line ends.
//   4. lg_finish: dq/dt = (r_0 + (r_1 + r_2)) / J, plus the source term if one is set.
// Volume flux variants ES-C, SF-KG and DC and the none / local Lax-Friedrichs interface dissipation
// are supported; the other optional terms of rhs_fix.cuh are not built at this degree.
#include <cuda_runtime.h>

#include "esdc_internal.h"
#include "flux_f64.cuh"
#include "kernels.h"
#include "rhs_fix.cuh"

namespace esdc {
namespace {

constexpr int LN = kLargeN;
constexpr int LN2 = LN * LN, LN3 = LN2 * LN;
constexpr int LT = LN / 2;               // threads per line in the pair rounds, one pair each
constexpr int LTHREADS = LN * LT;        // one plane: N lines
constexpr int VTHREADS = 256;
static_assert(32 % LT == 0, "the threads of a line must share a warp");

// Pair (i < j) handled by slot s in round r of the circle-method tournament over the N nodes of a
// line: node N-1 meets node r, and r + s meets r - s (mod N-1) for s = 1 .. N/2-1.  Over the N-1
// rounds every pair occurs once, and within a round every node occurs once.
__device__ __forceinline__ void round_pair(int r, int s, int& i, int& j) {
    int a, b;
    if (s == 0) {
        a = r;
        b = LN - 1;
    } else {
        a = r + s;
        if (a >= LN - 1) a -= LN - 1;
        b = r - s;
        if (b < 0) b += LN - 1;
    }
    i = a < b ? a : b;
    j = a < b ? b : a;
}

// Position i along its line and the line index t1 of entry k of a plane, chosen so that consecutive
// k are consecutive in memory (the line itself for l = 0, across lines for l = 1, 2).
__device__ __forceinline__ void plane_entry(int l, int k, int& i, int& t1) {
    if (l == 0) {
        i = k % LN;
        t1 = k / LN;
    } else {
        t1 = k % LN;
        i = k / LN;
    }
}

// Shared-memory index of node i of line t1 of a plane: the XOR keeps both a whole line (the pair loop) and node
// i of all lines (the line products) free of bank conflicts.
__device__ __forceinline__ int plane_slot(int t1, int i) { return t1 * LN + (i ^ t1); }

// ---- the float64 form of a plane: DC (whose pairs are sums of nodal fluxes), and planes out of the fixed-point
// range

// shared doubles: primitives 8 (hr, hu0..2, beta, qq, RT, c) | metric row l 3 | accumulators 5 | neighbours'
// entropy variables 4 x 32 | DC: nodal contravariant flux 5
template <int VF>
constexpr int plane_smem_doubles() {
    return (VF == kFluxDC ? 21 : 16) * LN2 + 4 * 2 * LN;
}

template <int VF>
__device__ __forceinline__ void plane_f64(double* sm, const double* __restrict__ q, const double* __restrict__ geom,
                                          const int32_t* __restrict__ nbr, const double* __restrict__ fnorm,
                                          double* __restrict__ rl, double* __restrict__ th, int64_t K,
                                          const OpsL& ops, const Phys& ph) {
    double* sPr = sm;
    double* sNm = sPr + 8 * LN2;
    double* sAc = sNm + 3 * LN2;
    double* sWn = sAc + 5 * LN2;
    [[maybe_unused]] double* sFl = sWn + 4 * 2 * LN;
    const int64_t b = blockIdx.x;
    const int64_t el = b / (3 * LN);
    const int rem = (int)(b - el * 3 * LN);
    const int l = rem / LN, t2 = rem - l * LN;
    const int st = dir_stride<LN>(l);
    const double* qe = q + el * 5 * LN3;

    for (int k = threadIdx.x; k < LN2; k += LTHREADS) {
        int i, t1;
        plane_entry(l, k, i, t1);
        const int node = line_base<LN>(l, t1, t2) + i * st;
        const int si = t1 * LN + i;
        double qv[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = qe[v * LN3 + node];
        Prim s;
        double RT, cs;
        to_prim(qv, ph, s, RT, cs);
        sPr[si] = s.hr;
        sPr[LN2 + si] = s.hu0;
        sPr[2 * LN2 + si] = s.hu1;
        sPr[3 * LN2 + si] = s.hu2;
        sPr[4 * LN2 + si] = s.beta;
        sPr[5 * LN2 + si] = s.qq;
        sPr[6 * LN2 + si] = RT;
        sPr[7 * LN2 + si] = cs;
        const double n0 = geom[(el * 10 + 1 + 3 * l) * LN3 + node];
        const double n1 = geom[(el * 10 + 2 + 3 * l) * LN3 + node];
        const double n2 = geom[(el * 10 + 3 + 3 * l) * LN3 + node];
        sNm[si] = n0;
        sNm[LN2 + si] = n1;
        sNm[2 * LN2 + si] = n2;
#pragma unroll
        for (int v = 0; v < 5; ++v) sAc[v * LN2 + si] = 0.0;
        if constexpr (VF == kFluxDC) {
            double f[5];
            euler_flux_prim(s, RT, n0, n1, n2, ph, f);
#pragma unroll
            for (int v = 0; v < 5; ++v) sFl[v * LN2 + si] = f[v];
        }
    }
    __syncthreads();

    const int line = threadIdx.x / LT, slot = threadIdx.x - (threadIdx.x / LT) * LT;
    const int lb = line * LN;
    for (int r = 0; r < LN - 1; ++r) {
        int i, j;
        round_pair(r, slot, i, j);
        const int ii = lb + i, jj = lb + j;
        double f[5];
        if constexpr (VF == kFluxDC) {
#pragma unroll
            for (int v = 0; v < 5; ++v) f[v] = sFl[v * LN2 + ii] + sFl[v * LN2 + jj];
        } else {
            Prim si, sj;
            load_prim(sPr, LN2, ii, si);
            load_prim(sPr, LN2, jj, sj);
            const double a0 = sNm[ii] + sNm[jj], a1 = sNm[LN2 + ii] + sNm[LN2 + jj],
                         a2 = sNm[2 * LN2 + ii] + sNm[2 * LN2 + jj];     // 2 x averaged metric
            if constexpr (VF == kFluxESC) ec_flux(si, sj, a0, a1, a2, ph, f);
            else kg_flux(si, sj, sPr[6 * LN2 + ii], sPr[6 * LN2 + jj], a0, a1, a2, ph, f);
        }
        const double c = ops.S[i][j];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            sAc[v * LN2 + ii] = fma(-c, f[v], sAc[v * LN2 + ii]);
            sAc[v * LN2 + jj] = fma(c, f[v], sAc[v * LN2 + jj]);
        }
        __syncwarp();
    }

    // interface SAT of the two faces normal to l at the line ends (slot 0: xi_l = -1, slot 1: +1)
    if (slot < 2) {
        const int side = slot;
        const int i = side ? LN - 1 : 0;
        const int lbase = line_base<LN>(l, line, t2);
        const int own = lbase + i * st;
        const int nbn = lbase + (side ? 0 : (LN - 1) * st);
        const int64_t nb = nbr[el * 6 + 2 * l + side];
        double qo[5], qn[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            qo[v] = qe[v * LN3 + own];
            qn[v] = q[nb * 5 * LN3 + v * LN3 + nbn];
        }
        const int si = lb + i;
        Prim so, sn;
        double RTn, cn;
        load_prim(sPr, LN2, si, so);
        to_prim(qn, ph, sn, RTn, cn);
        const double n0 = sNm[si], n1 = sNm[LN2 + si], n2 = sNm[2 * LN2 + si];
        double f[5];
        if constexpr (VF == kFluxESC) {
            ec_flux(so, sn, n0, n1, n2, ph, f);
        } else if constexpr (VF == kFluxKG) {
            kg_flux(so, sn, sPr[6 * LN2 + si], RTn, n0, n1, n2, ph, f);
        } else {
            double fo[5];
            euler_flux_prim(so, sPr[6 * LN2 + si], n0, n1, n2, ph, fo);
            euler_flux_prim(sn, RTn, n0, n1, n2, ph, f);
#pragma unroll
            for (int v = 0; v < 5; ++v) f[v] = 0.5 * (fo[v] + f[v]);
        }
        const double E = side ? 1.0 : -1.0;
        double lam = 0.0;
        if (ph.dissipation == 1) {
            const double nn = fnorm[(el * 6 + 2 * l + side) * LN2 + line + LN * t2];     // |n_J|
            const double lo = 2.0 * fabs(so.hu0 * n0 + so.hu1 * n1 + so.hu2 * n2) + sPr[7 * LN2 + si] * nn;
            const double ln = 2.0 * fabs(sn.hu0 * n0 + sn.hu1 * n1 + sn.hu2 * n2) + cn * nn;
            lam = 0.5 * fmax(lo, ln);
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) sAc[v * LN2 + si] += -E * f[v] - lam * (qo[v] - qn[v]);
        double* wn = sWn + side * LN + line;
        wn[0] = 4.0 * sn.beta * sn.hu0;
        wn[2 * LN] = 4.0 * sn.beta * sn.hu1;
        wn[4 * LN] = 4.0 * sn.beta * sn.hu2;
        wn[6 * LN] = -2.0 * sn.beta;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < LN2; k += LTHREADS) {      // entropy variables in place of hu and beta
        const double b4 = 4.0 * sPr[4 * LN2 + k];
#pragma unroll
        for (int m = 1; m < 4; ++m) sPr[m * LN2 + k] *= b4;
        sPr[4 * LN2 + k] = -0.5 * b4;
    }
    __syncthreads();

    double* out = rl + ((int64_t)l * K + el) * 5 * LN3;
    for (int k = threadIdx.x; k < LN2; k += LTHREADS) {
        int i, t1;
        plane_entry(l, k, i, t1);
        const int node = line_base<LN>(l, t1, t2) + i * st;
        const int si = t1 * LN + i;
#pragma unroll
        for (int v = 0; v < 5; ++v) out[v * LN3 + node] = sAc[v * LN2 + si] * ops.winv[i];
        if (ph.viscous) {
#pragma unroll 1
            for (int m = 0; m < 4; ++m) {
                const double* w = sPr + (1 + m) * LN2 + t1 * LN;
                double s = 0.0;
#pragma unroll
                for (int j = 0; j < LN; ++j) s += ops.D[i][j] * w[j];
                if (i == 0 || i == LN - 1) {
                    const int side = i != 0;
                    s += (side ? 0.5 : -0.5) * (sWn[m * 2 * LN + side * LN + t1] - w[i]) * ops.winv[i];
                }
                th[((el * 3 + l) * 4 + m) * LN3 + node] = s;
            }
        }
    }
}

template <int VF>
__global__ void __launch_bounds__(LTHREADS)
lg_volume(const double* __restrict__ q, const double* __restrict__ geom, const int32_t* __restrict__ nbr,
          const double* __restrict__ fnorm, double* __restrict__ rl, double* __restrict__ th, int64_t K,
          const __grid_constant__ OpsL ops, const __grid_constant__ Phys ph) {
    extern __shared__ double sm[];
    plane_f64<VF>(sm, q, geom, nbr, fnorm, rl, th, K, ops, ph);
}
template <int VF>
__device__ __noinline__ void plane_out_of_range(double* sm, const double* q, const double* geom, const int32_t* nbr,
                                                const double* fnorm, double* rl, double* th, int64_t K,
                                                const OpsL& ops, const Phys& ph) {
    plane_f64<VF>(sm, q, geom, nbr, fnorm, rl, th, K, ops, ph);
}

// ---- block fixed point

// out_i = sum_j D_ij v_j (units 2^kD) for the eight rows i of one half, in two partial sums of eight: the limb
// products of sixteen could leave 63 bits.  half is uniform in a warp, so the operator comes from the constant bank.
template <typename Store>
__device__ __forceinline__ void half_rows(const Fx (&v)[LN], const Fx (&D)[LN][LN], int half, Store store) {
#pragma unroll 1
    for (int r = 0; r < LN / 2; ++r) {
        const int i = half * (LN / 2) + r;
        long long o = 0;
#pragma unroll
        for (int c = 0; c < LN; c += LN / 2) {
            long long h = 0, m = kFxHalf + (LN / 2) * kFxLow;
#pragma unroll
            for (int j = c; j < c + LN / 2; ++j) fx_mac(h, m, D[i][j], v[j]);
            o += h + (m >> 30);
        }
        store(i, o);
    }
}

// Line products of a plane: thread t takes variable `var`, line `line`, rows of half `half`
struct LineTask {
    int half, var, line;
    __device__ __forceinline__ explicit LineTask(int t) : half(t >> 6), var((t >> 4) & 3), line(t & (LN - 1)) {}
};

// shared doubles of lg_volume_fix: pair inputs NP | metric 3 | theta, then results 5, each [N^2] | neighbours'
// pair inputs and sound speed (NP + 1) x 32 | face terms 5 x 32
template <int VF>
constexpr int fix_inputs() {
    return VF == kFluxESC ? 6 : 7;
}
template <int VF>
constexpr int fix_smem_doubles() {
    constexpr int NP = fix_inputs<VF>(), need = (NP + 8) * LN2 + (NP + 6) * 2 * LN;
    return need > plane_smem_doubles<VF>() ? need : plane_smem_doubles<VF>();
}

// ES-C and SF-KG, a plane's nodes and their neighbours' face nodes under common exponents; a plane out of the
// fixed-point range takes the float64 form.  In the pair loop a warp holds two lines: at cyclic distance k =
// 1..N/2 the lane of node i evaluates the pair (i, i + k mod N), S_ij f is summed in registers on one side and
// by a shuffle on the other.  One warp evaluates the 32 face terms while the others begin on the lines, which a
// counter hands out; which warp, changes with the plane.
// The sums over a line stay inside 63 bits by the bounds at fix_scale.
// In float64 the pairs kept that pipe (64 clocks per instruction and scheduler) busy; bound now by the multiply
// and shift pipes and their latency.  Viscous ES-C residual of the Taylor-Green flow on 6 x 5 x 7 elements, with
// theta from here and the divergence's line products in fixed point too: 3.89 -> 1.00 ms, of which this kernel
// 0.64, lg_viscous 0.21 (the float64 pipe), lg_visc_div 0.14.  Four / five / six CTAs per SM on 6^3 elements:
// 1.004 / 0.996 / 0.988 ms.
template <int VF>
__global__ void __launch_bounds__(LTHREADS, 6)
lg_volume_fix(const double* __restrict__ q, const double* __restrict__ geom, const int32_t* __restrict__ nbr,
              const double* __restrict__ fnorm, double* __restrict__ rl, double* __restrict__ th, int64_t K,
              const __grid_constant__ OpsL ops, const __grid_constant__ Phys ph, const int32_t* __restrict__ kn) {
    constexpr int NP = fix_inputs<VF>(), NE = VF == kFluxESC ? 10 : 12, NF = 2 * LN;
    extern __shared__ double sm[];
    __shared__ int sE[NE], sNext;
    __shared__ FixScale sScale;
    __shared__ Fx sS[LT * LN];
    double* sNm = sm + NP * LN2;
    double* sAc = sNm + 3 * LN2;
    double* sNb = sAc + 5 * LN2;
    double* sFc = sNb + (NP + 1) * NF;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t b = blockIdx.x;
    const int64_t el = b / (3 * LN);
    const int rem = (int)(b - el * 3 * LN);
    const int l = rem / LN, t2 = rem - l * LN;
    const int st = dir_stride<LN>(l);
    const double* qe = q + el * 5 * LN3;
    // the face warp: lane = (side, line)
    const bool fw = warp == (int)(b & (LTHREADS / 32 - 1));
    const int side = lane / LN, fline = lane % LN;
    const int fbase = line_base<LN>(l, fline, t2);
    const int own = fbase + (side ? LN - 1 : 0) * st;
    const int64_t nb = nbr[el * 6 + 2 * l + side];
    const double* qn = q + nb * 5 * LN3 + fbase + (side ? 0 : (LN - 1) * st);
    if (t < NE) sE[t] = 0;
    if (t == 0) sNext = 0;
    for (int k = t; k < LT * LN; k += LTHREADS) sS[k] = ops.SF[k / LN][k % LN];
    __syncthreads();

    int E[NE] = {};
#pragma unroll
    for (int h = 0; h < LN2 / LTHREADS; ++h) {
        int i, t1;
        plane_entry(l, t + h * LTHREADS, i, t1);
        const int node = line_base<LN>(l, t1, t2) + i * st;
        const int si = plane_slot(t1, i);
        double qv[5], RT, pi[NP];
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = qe[v * LN3 + node];
        int En[NE] = {};
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const double g = geom[(el * 10 + 1 + 3 * l + m) * LN3 + node];
            sNm[m * LN2 + si] = g;
            E[5] = max(E[5], biased_exp(g));
        }
        pair_inputs<VF>(qv, ph, pi, RT);
#pragma unroll
        for (int m = 0; m < NP; ++m) sm[m * LN2 + si] = pi[m];
        rhs_exponents(pi, En);
#pragma unroll
        for (int m = 0; m < NE; ++m) E[m] = max(E[m], En[m]);
    }
    if (fw) {
        double qv[5], RT, pi[NP];
        int En[NE] = {};
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = qn[v * LN3];
        pair_inputs<VF>(qv, ph, pi, RT);
#pragma unroll
        for (int m = 0; m < NP; ++m) sNb[m * NF + lane] = pi[m];
        sNb[NP * NF + lane] = sqrt_newton(ph.gamma * RT);
        rhs_exponents(pi, En);
#pragma unroll
        for (int m = 0; m < NE; ++m) E[m] = max(E[m], En[m]);
    }
    block_max<true>(sE, 0, E, lane);
    __syncthreads();
    if (kn[el] == kStretched || !rhs_range_ok(sE, 3)) {
        __syncthreads();
        plane_out_of_range<VF>(sm, q, geom, nbr, fnorm, rl, th, K, ops, ph);
        return;
    }
    {
        int Es[NE];
#pragma unroll
        for (int m = 0; m < NE; ++m) Es[m] = sE[m];
        const FixScale s = element_scale<VF>(Es, ops.kg);
        if (t == 0) sScale = s;
#pragma unroll
        for (int h = 0; h < LN2 / LTHREADS; ++h) {
            int i, t1;
            plane_entry(l, t + h * LTHREADS, i, t1);
            const int si = plane_slot(t1, i);
            scale_inputs<VF>(sm + si, reinterpret_cast<Fx*>(sm) + si, LN2, s);
#pragma unroll
            for (int m = 0; m < 3; ++m)
                reinterpret_cast<Fx*>(sNm)[m * LN2 + si] = fx_split(fx_from_double(sNm[m * LN2 + si], s.kn));
        }
        if (fw) scale_inputs<VF>(sNb + lane, reinterpret_cast<Fx*>(sNb) + lane, NF, s);
    }
    __syncthreads();
    const Fx* XP = reinterpret_cast<const Fx*>(sm);
    const Fx* XN = reinterpret_cast<const Fx*>(sNm);
    const Fx* XB = reinterpret_cast<const Fx*>(sNb);
    const FixScale& s = sScale;

    // theta_l = D_l w + E/2 (w_nbr - w)/w_i at the line ends: w2..w4 = 2 beta u in units 2^(kb + ku), beta for
    // w5 = -2 beta
    if (ph.viscous) {
        const LineTask lt(t);
        const Fx* B = XP + 4 * LN2;
        const Fx* U = XP + (1 + (lt.var < 3 ? lt.var : 0)) * LN2;
        Fx v[LN];
#pragma unroll
        for (int j = 0; j < LN; ++j) {
            const int k = plane_slot(lt.line, j);
            v[j] = lt.var < 3 ? fx_split(fx_mul(B[k], U[k]) * 4) : B[k];
        }
        const Fx* g = XB + lt.half * LN + lt.line;
        const Fx wn = lt.var < 3 ? fx_split(fx_mul(g[4 * NF], g[(1 + lt.var) * NF]) * 4) : g[4 * NF];
        const Fx wo = lt.half ? v[LN - 1] : v[0];
        const long long lift = fx_mul<0>(ops.LF, lt.half ? fx_sub(wn, wo) : fx_sub(wo, wn));
        const int end = lt.half ? LN - 1 : 0, ku = ops.kD + s.kb + (lt.var < 3 ? s.ku : 1);
        double* T = sAc + lt.var * LN2;
        half_rows(v, ops.DF, lt.half, [&](int i, long long o) {
            const double x = fx_to_double(i == end ? o + lift : o, ku);
            T[plane_slot(lt.line, i)] = lt.var < 3 ? x : -x;
        });
        __syncthreads();
#pragma unroll
        for (int h = 0; h < LN2 / LTHREADS; ++h) {
            int i, t1;
            plane_entry(l, t + h * LTHREADS, i, t1);
            double* out = th + (el * 3 + l) * 4 * LN3 + line_base<LN>(l, t1, t2) + i * st;
#pragma unroll
            for (int k = 0; k < 4; ++k) out[k * LN3] = sAc[k * LN2 + plane_slot(t1, i)];
        }
        __syncthreads();
    }

    // interface SAT: -(E f_2pt(own, nbr).n_J + lambda/2 (q_own - q_nbr)) / w_i
    if (fw) {
        const int os = plane_slot(fline, side ? LN - 1 : 0);
        const PrimFx a = load_inputs<VF>(XP + os, LN2), c = load_inputs<VF>(XB + lane, NF);
        const Fx n0 = XN[os], n1 = XN[LN2 + os], n2 = XN[2 * LN2 + os];
        long long f[5];
        two_point<VF>(a, c, n0, n1, n2, ops.CG, ph.inv_gm1, s, f);
        double qo[5], lam = 0.0;
        if (ph.dissipation == 1) {
            Prim so;
            double RT;
#pragma unroll
            for (int v = 0; v < 5; ++v) qo[v] = qe[v * LN3 + own];
            to_prim_fx(qo, ph, so, RT);
            const double nn = fnorm[(el * 6 + 2 * l + side) * LN2 + fline + LN * t2];     // |n_J|
            const double co = sqrt_newton(ph.gamma * RT), cn = sNb[NP * NF + lane];
            const double uo = fx_to_double(fx_dot(a.u0, n0, a.u1, n1, a.u2, n2), s.ku + s.kn + 1);
            const double un = fx_to_double(fx_dot(c.u0, n0, c.u1, n1, c.u2, n2), s.ku + s.kn + 1);
            lam = ops.winv[0] * (0.5 * fmax(fma(co, nn, fabs(uo)), fma(cn, nn, fabs(un))));
        }
        const double wi = side ? -ops.winv[LN - 1] : ops.winv[0];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double r = wi * fx_to_double(f[v], v == 0 ? s.k0 : (v == 4 ? s.k5 : s.km));
            if (ph.dissipation == 1) r = fma(-lam, qo[v] - qn[v * LN3], r);
            sFc[v * NF + lane] = r;
        }
    }

    const int i = lane % LN;
    const double w = ops.winv[i];
    for (;;) {
        int task = 0;
        if (lane == 0) task = atomicAdd(&sNext, 1);
        task = __shfl_sync(0xffffffffu, task, 0);
        if (task >= LN / 2) break;
        const int line = 2 * task + lane / LN, ii = plane_slot(line, i);
        const PrimFx a = load_inputs<VF>(XP + ii, LN2);
        const Fx na0 = XN[ii], na1 = XN[LN2 + ii], na2 = XN[2 * LN2 + ii];
        unsigned long long acc[5] = {0, 0, 0, 0, 0};
#pragma unroll 1
        for (int k = 1; k <= LT; ++k) {
            long long Pv[5] = {0, 0, 0, 0, 0};
            if (2 * k < LN || i < k) {
                const int jj = plane_slot(line, (i + k) & (LN - 1));
                const PrimFx c = load_inputs<VF>(XP + jj, LN2);
                const Fx S = sS[(k - 1) * LN + i];
                const Fx n0 = fx_split(fx_mul<2>(S, fx_add(na0, XN[jj]))), n1 = fx_split(fx_mul<2>(S, fx_add(na1, XN[LN2 + jj]))),
                         n2 = fx_split(fx_mul<2>(S, fx_add(na2, XN[2 * LN2 + jj])));
                two_point<VF>(a, c, n0, n1, n2, ops.CG, ph.inv_gm1, s, Pv);
#pragma unroll
                for (int v = 0; v < 5; ++v) acc[v] -= (unsigned long long)Pv[v];
            }
            const int from = (lane & ~(LN - 1)) + ((i - k) & (LN - 1));
#pragma unroll
            for (int v = 0; v < 5; ++v) acc[v] += (unsigned long long)__shfl_sync(0xffffffffu, Pv[v], from);
        }
#pragma unroll
        for (int v = 0; v < 5; ++v)
            sAc[v * LN2 + ii] = w * fx_to_double((long long)acc[v], v == 0 ? s.k0 : (v == 4 ? s.k5 : s.km));
    }
    __syncthreads();

    double* out = rl + ((int64_t)l * K + el) * 5 * LN3;
#pragma unroll
    for (int h = 0; h < LN2 / LTHREADS; ++h) {
        int i, t1;
        plane_entry(l, t + h * LTHREADS, i, t1);
        const int node = line_base<LN>(l, t1, t2) + i * st;
        const int si = plane_slot(t1, i);
        const bool end = i == 0 || i == LN - 1;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double r = sAc[v * LN2 + si];
            if (end) r += sFc[v * NF + (i ? LN : 0) + t1];
            out[v * LN3 + node] = r;
        }
    }
}

// Viscous fluxes, one thread per node: th holds theta_a[k] on entry; g_m = J^-1 sum_a Ja_am theta_a, then tau, the
// heat flux and Ftilde_l = sum_m Ja_lm F^V_m (eq. Fv, eq. tau), written over theta and, on the faces of direction
// l, to the trace buffer.  J^-1 goes into the two coefficients mu RT/J and (kappa/R) RT^2/J.
__global__ void __launch_bounds__(VTHREADS)
lg_viscous(const double* __restrict__ q, const double* __restrict__ geom, const double* __restrict__ jinv,
           double* __restrict__ th, double* __restrict__ trace, int64_t K, const Phys ph) {
    const int64_t n = K * LN3, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t gn = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gn < n; gn += stride) {
        const int64_t el = gn / LN3;
        const int node = (int)(gn - el * LN3);
        const int i1 = node % LN, i2 = (node / LN) % LN, i3 = node / LN2;
        double* te = th + el * 12 * LN3 + node;
        const double* G = geom + el * 10 * LN3 + node;
        double Ja[3][3];
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
            for (int m = 0; m < 3; ++m) Ja[l][m] = G[(1 + 3 * l + m) * LN3];
        double g[3][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double t0 = te[k * LN3], t1 = te[(4 + k) * LN3], t2 = te[(8 + k) * LN3];
#pragma unroll
            for (int m = 0; m < 3; ++m) g[m][k] = fma(Ja[2][m], t2, fma(Ja[1][m], t1, Ja[0][m] * t0));
        }
        double qv[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = q[(el * 5 + v) * LN3 + node];
        Prim s;
        double RT;
        to_prim_fx(qv, ph, s, RT);
        const double Jinv = jinv[gn];
        const double y = ph.mu * RT * Jinv, z = ph.kappa_R * RT * RT * Jinv;
        const double u[3] = {2.0 * s.hu0, 2.0 * s.hu1, 2.0 * s.hu2};
        // du_k/dx_m = RT (g_m[k] + u_k g_m[3]); dT/dx_m = (RT)^2/R g_m[3]
        double du[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < 3; ++m) du[k][m] = fma(u[k], g[m][3], g[m][k]);
        const double div3 = (2.0 / 3.0) * (du[0][0] + du[1][1] + du[2][2]);
        double FV[3][4];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
#pragma unroll
            for (int i = 0; i <= m; ++i) {
                FV[m][i] = y * (i == m ? fma(2.0, du[i][i], -div3) : du[i][m] + du[m][i]);
                FV[i][m] = FV[m][i];
            }
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) FV[m][3] = fma(FV[m][0], u[0], fma(FV[m][1], u[1], fma(FV[m][2], u[2], z * g[m][3])));
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            double Ft[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) Ft[k] = fma(Ja[l][2], FV[2][k], fma(Ja[l][1], FV[1][k], Ja[l][0] * FV[0][k]));
#pragma unroll
            for (int k = 0; k < 4; ++k) te[(4 * l + k) * LN3] = Ft[k];
            const int il = l == 0 ? i1 : (l == 1 ? i2 : i3);
            if (il == 0 || il == LN - 1) {
                const int side = il == LN - 1;
                const int fi = l == 0 ? (i2 + LN * i3) : (l == 1 ? (i1 + LN * i3) : (i1 + LN * i2));
                double* tr = trace + ((el * 6 + 2 * l + side) * 4) * LN2 + fi;
#pragma unroll
                for (int k = 0; k < 4; ++k) tr[k * LN2] = Ft[k];
            }
        }
    }
}

// r_l += D_l Ftilde_l along the lines of one plane, plus the BR1 interface term at the line ends.  The line
// products in fixed point under the plane's largest exponents (momentum, energy), or in float64 where those are
// not far inside its range.
__global__ void __launch_bounds__(LTHREADS)
lg_visc_div(const double* __restrict__ ft, const double* __restrict__ trace, const int32_t* __restrict__ nbr,
            double* __restrict__ rl, int64_t K, const __grid_constant__ OpsL ops) {
    __shared__ double sF[4 * LN2];
    __shared__ int sE[2];
    const int t = threadIdx.x, lane = t & 31;
    const int64_t b = blockIdx.x;
    const int64_t el = b / (3 * LN);
    const int rem = (int)(b - el * 3 * LN);
    const int l = rem / LN, t2 = rem - l * LN;
    const int st = dir_stride<LN>(l);
    constexpr int EN = LN2 / LTHREADS;
    if (t < 2) sE[t] = 0;
    __syncthreads();
    double f[EN][4];
    int E[2] = {0, 0};
#pragma unroll
    for (int h = 0; h < EN; ++h) {
        int i, t1;
        plane_entry(l, t + h * LTHREADS, i, t1);
        const double* p = ft + (el * 3 + l) * 4 * LN3 + line_base<LN>(l, t1, t2) + i * st;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[h][k] = p[k * LN3];
            E[k == 3] = max(E[k == 3], biased_exp(f[h][k]));
            sF[k * LN2 + plane_slot(t1, i)] = f[h][k];
        }
    }
    block_max<true>(sE, 0, E, lane);
    __syncthreads();
    const LineTask lt(t);
    if (max(sE[0], sE[1]) < 1900) {
        const int k = sE[lt.var == 3] - 1021;
        Fx v[LN];
#pragma unroll
        for (int j = 0; j < LN; ++j) v[j] = fx_split(fx_from_double(sF[lt.var * LN2 + plane_slot(lt.line, j)], k));
        __syncthreads();
        half_rows(v, ops.DF, lt.half, [&](int i, long long o) {
            sF[lt.var * LN2 + plane_slot(lt.line, i)] = fx_to_double(o, ops.kD + k);
        });
    } else {
        double v[LN];
#pragma unroll
        for (int j = 0; j < LN; ++j) v[j] = sF[lt.var * LN2 + plane_slot(lt.line, j)];
        __syncthreads();
        for (int r = 0; r < LN / 2; ++r) {
            const int i = lt.half * (LN / 2) + r;
            double o = 0.0;
#pragma unroll
            for (int j = 0; j < LN; ++j) o += ops.D[i][j] * v[j];
            sF[lt.var * LN2 + plane_slot(lt.line, i)] = o;
        }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < EN; ++h) {
        int i, t1;
        plane_entry(l, t + h * LTHREADS, i, t1);
        double* out = rl + (((int64_t)l * K + el) * 5 + 1) * LN3 + line_base<LN>(l, t1, t2) + i * st;
        const bool end = i == 0 || i == LN - 1;
        const int side = i != 0;
        const int64_t nb = end ? nbr[el * 6 + 2 * l + side] : 0;
        const double* tn = trace + ((nb * 6 + 2 * l + 1 - side) * 4) * LN2 + t1 + LN * t2;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double d = sF[k * LN2 + plane_slot(t1, i)];
            if (end) d += (side ? 0.5 : -0.5) * (tn[k * LN2] - f[h][k]) * ops.winv[i];
            out[k * LN3] += d;
        }
    }
}

// dq/dt = (r_0 + (r_1 + r_2)) / J, one thread per node.
__global__ void __launch_bounds__(256)
lg_finish(const double* __restrict__ rl, const double* __restrict__ jinv, double* __restrict__ dqdt, int64_t K,
          const double* __restrict__ src) {
    const int64_t n = K * LN3, part = K * 5 * LN3;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += stride) {
        const int64_t el = g / LN3;
        const int node = (int)(g - el * LN3);
        const double Jinv = jinv[g];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            const int64_t i = (el * 5 + v) * LN3 + node;
            const double r = (rl[i] + (rl[part + i] + rl[2 * part + i])) * Jinv;
            dqdt[i] = src ? r + src[i] : r;
        }
    }
}

template <int VF>
cudaError_t launch_volume(const esdc_ctx* c, const double* q, cudaStream_t s) {
    const unsigned grid = (unsigned)(c->K * 3 * LN);
    if (VF == kFluxDC || c->float64_form) {
        lg_volume<VF><<<grid, LTHREADS, plane_smem_doubles<VF>() * sizeof(double), s>>>(
            q, c->d_geom, c->d_nbr, c->d_fnorm, c->d_lr, c->d_lft, c->K, c->opsl, c->phys);
        return cudaGetLastError();
    }
    if constexpr (VF != kFluxDC)
        lg_volume_fix<VF><<<grid, LTHREADS, fix_smem_doubles<VF>() * sizeof(double), s>>>(
            q, c->d_geom, c->d_nbr, c->d_fnorm, c->d_lr, c->d_lft, c->K, c->opsl, c->phys, c->d_kn);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rhs_large(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    if (c->N != LN || !c->d_lr || !c->d_lft) return cudaErrorInvalidValue;
    if (ev) cudaEventRecord(ev[0], s);
    cudaError_t e;
    switch (c->setup.volume_flux) {
        case kFluxESC: e = launch_volume<kFluxESC>(c, q, s); break;
        case kFluxKG: e = launch_volume<kFluxKG>(c, q, s); break;
        case kFluxDC: e = launch_volume<kFluxDC>(c, q, s); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    int64_t blocks = (c->n_nodes + 255) / 256;
    if (blocks > grid_cap()) blocks = grid_cap();
    if (c->phys.viscous) {
        lg_viscous<<<(unsigned)blocks, VTHREADS, 0, s>>>(q, c->d_geom, c->d_jinv, c->d_lft, (double*)c->d_trace, c->K,
                                                         c->phys);
        lg_visc_div<<<(unsigned)(c->K * 3 * LN), LTHREADS, 0, s>>>(c->d_lft, (const double*)c->d_trace, c->d_nbr, c->d_lr,
                                                                  c->K, c->opsl);
    }
    lg_finish<<<(unsigned)blocks, 256, 0, s>>>(c->d_lr, c->d_jinv, dqdt, c->K, c->d_src);
    if (ev) {
        cudaEventRecord(ev[1], s);
        cudaEventRecord(ev[2], s);
        cudaEventRecord(ev[3], s);
    }
    return cudaGetLastError();
}

}  // namespace esdc
