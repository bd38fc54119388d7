// Residual of the float64 form in block fixed point (fix_f64.cuh): flux differencing with the
// Chandrashekar flux (ES-C, eq. discEL), the Kennedy-Gruber flux (SF-KG) or the nodal fluxes (DC), the
// interface SAT, BR1 entropy-variable gradients, viscous fluxes and their divergence (eq. MacroForm,
// eq. NSL) for p <= 7.  rhs_fix_*.cu instantiate it.
//
// One element per group of N^3 threads (EPB elements per CTA).  Float64 is kept where it is needed or
// cheap: primitives of own and neighbour states, the dissipation of the interface term, the sum of the
// directions' results, the scaling by 1/J and everything in global memory.  Phases:
//   0. primitives of the nodes and of the neighbours' face nodes; the element's largest and smallest
//      exponents; everything scaled to Q60 limbs in shared memory.  An element out of the fixed-point
//      range sends its CTA to the float64 form (element_f64.cuh).
//   1. volume: one thread per (node, direction), whole lines side by side in a warp.  At cyclic distance
//      k = 1..N/2 the thread of node i evaluates the pair (i, i + k mod N), so that each pair is
//      evaluated once; S_ij f is summed in registers on one side and by a shuffle on the other.  DC: the
//      nodal contravariant fluxes per node in float64, then one thread per line and variable, each line in
//      fixed point under its own largest exponent.
//   2. interface: one thread per face node; two-point flux in fixed point (DC: float64), dissipation in float64.
//   3. viscous: lines of w for theta_a = D_a w + lift (one thread per line and variable, the operator
//      from the constant bank), one thread per node for the fluxes, lines again for the divergence.
//
// Bound: multiply (8 lanes per clock and scheduler for a 32 x 32 -> 64 product) and shift/logic (16) pipes
// in phases 1 and 3, the float64 pipe (half a lane) in 0 and 2.  Against the all-float64 kernel, which
// kept the float64 pipe 87% busy, per viscous residual of the Taylor-Green flow: 8.59 -> 2.92 ms at p = 7
// on 20^3 elements, 0.92 -> 0.31 ms at p = 4 on 16^3, 2.58 -> 1.00 ms at p = 2 on 41 x 37 x 39.  Its error
// against extended precision, worst variable over flows along one axis and all, is 0.6 to 1.04 of the float64
// kernel's (kMaxStretch, fix_speed_ok; DC's energy at Mach 2 1.12).
#pragma once

#include <cuda_runtime.h>

#include "element_f64.cuh"
#include "esdc_internal.h"
#include "fix_f64.cuh"
#include "kernels.h"
#include "visc_sat.cuh"

namespace esdc {
namespace {

// Node slots of the limb arrays: rows of S2, layers of S3 (see slot).
template <int N>
struct FixSlot {
    static constexpr bool PAD = N == 4 || N == 6;
    static constexpr int S2 = PAD ? N + 1 : N, S3 = N * S2 + (PAD ? 1 : 0), SL = N * S3;
};

// WIDE: one element per CTA on as many warps as its pair loop has tasks (N = 7: half as many), for meshes
// that leave SMs idle otherwise: what counts there is the length of one element's chain.
template <int N, int VF, bool WIDE = false>
struct FixCfg {
    static constexpr int N2 = N * N, N3 = N * N * N;
    static constexpr int EPB = WIDE ? 1 : Cfg<N>::EPB;
    // Whole warps (the pair loop's shuffles); N = 6 one more than its nodes fill, which makes its 24 pair
    // tasks three rounds (2.43 -> 2.34 ms on 26^3 elements)
    static constexpr int THREADS = WIDE ? (N == 2 ? 96 : (N == 3 ? 128 : (N == 4 ? 192 : (N == 5 ? 480 : 640))))
                                        : (N == 6 ? 256 : (EPB * N3 + 31) / 32 * 32);
    static constexpr int WARPS = THREADS / 32;
    // Resident CTAs the registers are capped for: as many as the shared memory lets in.  The kernel takes
    // 124 to 174 registers left alone; the few spills cost less than the warps bring (N = 7, two CTAs
    // instead of one: 3.01 -> 2.39 ms on 22^3; N = 5, five instead of four: 2.31 -> 2.29 ms on 32^3; N = 3:
    // 1.10 -> 1.07 ms on 40^3; N = 2 with five: 1.48 -> 1.51 ms, so four; N = 8 with 24 or 20 warps on its
    // one CTA: 2.92 -> 2.96 and 3.01 ms on 20^3, so 16)
    static constexpr int MINB = WIDE || N == 8 ? 1 : (N >= 6 ? 2 : (N == 5 || N == 3 ? 5 : 4));
    // pair loop: LPW whole lines per warp, TPD warp tasks per direction
    static constexpr int LPW = 32 / N, TPD = (EPB * N2 + LPW - 1) / LPW;
    static constexpr int SL = FixSlot<N>::SL;
    // shared memory per element in 8-byte units
    static constexpr int XN = 0;                 // [9][SL] metric rows; later the viscous fluxes' momentum part
    static constexpr int NP = VF == kFluxESC ? 6 : 7;
    static constexpr int XP = 9 * SL;            // [NP][SL] pair inputs (PrimFx); later [3][SL] the viscous
                                                 //          fluxes' energy part
    static constexpr int XW = XP + NP * SL;      // [3][SL] w2..w4 = 2 beta u
    static constexpr int R = XW + 3 * SL;        // [3][5][SL] results per direction (float64; DC: the nodal
                                                 //            fluxes before); then [12][SL] theta
    static constexpr int P = R + 15 * SL;        // [N3] float64 RT
    static constexpr int F = P + N3;             // [NP + 1][6 N2] neighbour face nodes: pair inputs, sound speed
    static constexpr int SM = F + (NP + 1) * 6 * N2;
};

// Slot of node (i1, i2, i3) in the limb arrays.  A half-warp of 64-bit loads covers two lines of eight
// nodes at N = 8: the XOR spreads every direction's over all banks without padding; N = 4 and 6 take
// odd row strides; odd N needs nothing.
template <int N>
__device__ __forceinline__ int slot(int i1, int i2, int i3) {
    if constexpr (N == 8) return (i1 ^ (2 * ((i2 >> 1) ^ (i3 >> 1)))) + 8 * (i2 ^ (i3 & 1)) + 64 * i3;
    else return i1 + FixSlot<N>::S2 * i2 + FixSlot<N>::S3 * i3;
}
// node i of line (c1, c2) of direction l
template <int N>
__device__ __forceinline__ int line_slot(int l, int i, int c1, int c2) {
    return l == 0 ? slot<N>(i, c1, c2) : (l == 1 ? slot<N>(c1, i, c2) : slot<N>(c1, c2, i));
}

// Element-wide maxima of NV non-negative integers into out (element e's, shared memory, zeroed).  Called by
// the active threads of a warp; UNIFORM: of one element.  The lanes of an element reduce first.
template <bool UNIFORM, int NV>
__device__ __forceinline__ void block_max(int* out, int e, int (&v)[NV], int lane) {
    unsigned mask = __activemask();
    if constexpr (!UNIFORM) mask = __match_any_sync(mask, e);
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = __reduce_max_sync(mask, v[i]);
    if (lane == __ffs(mask) - 1)
#pragma unroll
        for (int i = 0; i < NV; ++i) atomicMax(out + i, v[i]);
}

// Logarithmic means beyond the series of ec_flux_fx, in float64 from the fixed-point inputs.
__device__ __noinline__ long long log_mean_f64(long long a, long long b, int k, double num, int kout) {
    const double x = fx_to_double(a, k), y = fx_to_double(b, k), lg = log(x / y);
    return fx_from_double(num > 0.0 ? 0.5 * num * lg / (x - y) : 2.0 * (x - y) / lg, kout);
}
struct LogMeanF64 {
    Fx ra, rb, ba, bb;
    const FixScale& s;
    double inv_gm1;
    __device__ __forceinline__ long long rho() const { return log_mean_f64(fx_join(ra), fx_join(rb), s.kr, 0.0, s.kr); }
    __device__ __forceinline__ long long inv_beta() const {
        return log_mean_f64(fx_join(ba), fx_join(bb), s.kb, inv_gm1, s.kA);
    }
};

// Primitives as in to_prim, with the float64 operations that can go to the integer pipe there: halving
// is an exponent decrement (zeros, infinities and NaNs end up out of the fixed-point range).
__device__ __forceinline__ double half_of(double x) { return __hiloint2double(__double2hiint(x) - (1 << 20), __double2loint(x)); }
__device__ __forceinline__ void to_prim_fx(const double* q, const Phys& ph, Prim& s, double& RT) {
    const double ri = rcp_cubic(q[0]), rh = half_of(ri);
    s.hu0 = q[1] * rh;
    s.hu1 = q[2] * rh;
    s.hu2 = q[3] * rh;
    s.qq = fma(s.hu2, s.hu2, fma(s.hu1, s.hu1, s.hu0 * s.hu0));
    const double p = ph.gm1 * fma(-2.0 * q[0], s.qq, q[4]);
    s.hr = half_of(q[0]);
    s.beta = s.hr * rcp_cubic(p);
    RT = p * ri;
}
// The pair loop's inputs of a node, in PrimFx's order: half density, half velocity, beta, then |u|^2/4
// (ES-C); or the node's part of the mean specific energy and half the pressure (SF-KG); or the specific
// enthalpy and half the pressure (DC).
template <int VF, int NP>
__device__ __forceinline__ void pair_inputs(const double* q, const Phys& ph, double (&pi)[NP], double& RT) {
    Prim s;
    to_prim_fx(q, ph, s, RT);
    pi[0] = s.hr;
    pi[1] = s.hu0;
    pi[2] = s.hu1;
    pi[3] = s.hu2;
    pi[4] = s.beta;
    if constexpr (VF == kFluxESC) pi[5] = s.qq;
    else {
        pi[5] = VF == kFluxKG ? fma(0.5 * ph.inv_gm1, RT, s.qq) : fma(ph.gamma * ph.inv_gm1, RT, 2.0 * s.qq);
        pi[6] = s.hr * RT;
    }
}
// Exponents of a node's pair inputs for the element-wide maxima; a sign bit counts as out of range (density
// and beta must be positive).
template <int NP, int NE>
__device__ __forceinline__ void pair_exponents(const double (&pi)[NP], int (&E)[NE]) {
    E[0] = (unsigned)double_hi(pi[0]) >> 20;
    E[1] = 4096 - E[0];
    E[2] = max(biased_exp(pi[1]), max(biased_exp(pi[2]), biased_exp(pi[3])));
    E[3] = (unsigned)double_hi(pi[4]) >> 20;
    E[4] = 4096 - E[3];
}
// The same for the residual kernels: the velocity components' speed codes apart (E[2], E[8], E[9]), and SF-KG's last
// two inputs.
template <int NP, int NE>
__device__ __forceinline__ void rhs_exponents(const double (&pi)[NP], int (&E)[NE]) {
    pair_exponents(pi, E);
    E[2] = speed_code(pi[1]);
    E[8] = speed_code(pi[2]);
    E[9] = speed_code(pi[3]);
    if constexpr (NE == 12) {
        E[10] = biased_exp(pi[5]);
        E[11] = biased_exp(pi[6]);
    }
}
template <int NE>
__device__ __forceinline__ bool rhs_range_ok(const int (&E)[NE], int most_speed = 5) {
    return fix_range_ok(E[0], 4096 - E[1], speed_exponent(E[2], E[8], E[9]), E[3], 4096 - E[4], E[5]) &&
           fix_speed_ok(E[2], E[8], E[9], 4096 - E[4], most_speed) && E[6] < 1151 && E[7] < 1151;
}
// the element's scales from its maxima
template <int VF, int NE>
__device__ __forceinline__ FixScale element_scale(const int (&E)[NE], int kg) {
    const int Eu = speed_exponent(E[2], E[8], E[9]);
    if constexpr (VF == kFluxESC) return fix_scale(E[0], 4096 - E[1], Eu, E[3], 4096 - E[4], E[5], E[6], E[7], kg);
    else if constexpr (VF == kFluxKG) return fix_scale_kg(E[0], Eu, E[3], E[5], E[6], E[7], E[10], E[11]);
    else return fix_scale_dc(Eu, E[3], E[5], E[6], E[7]);
}
// a node's (or neighbour's) pair inputs from float64 to limbs, arrays `stride` apart; of DC's only those of the
// viscous terms
template <int VF>
__device__ __forceinline__ void scale_inputs(const double* p, Fx* x, int stride, const FixScale& s) {
#pragma unroll
    for (int m = 1; m < 4; ++m) x[m * stride] = fx_split(fx_from_double(p[m * stride], s.ku));
    x[4 * stride] = fx_split(fx_from_double(p[4 * stride], s.kb));
    if constexpr (VF == kFluxDC) return;
    x[0] = fx_split(fx_from_double(p[0], s.kr));
    x[5 * stride] = fx_split(fx_from_double(p[5 * stride], s.kq));
    if constexpr (VF != kFluxESC) x[6 * stride] = fx_split(fx_from_double(p[6 * stride], s.kp));
}
template <int VF>
__device__ __forceinline__ PrimFx load_inputs(const Fx* x, int stride) {
    PrimFx a = {x[0], x[stride], x[2 * stride], x[3 * stride], x[4 * stride], x[5 * stride], Fx{0, 0}};
    if constexpr (VF != kFluxESC) a.p = x[6 * stride];
    return a;
}

// The elements of a CTA left to the float64 form; out of line, so that the kernel's registers are its own.  With
// every element out of range a residual takes phase 0 more than the all-float64 kernel did: ES-C p = 1 1.08 against
// 1.00 ms on 40^3, p = 3 1.84 against 1.81 on 24^3, p = 4 1.57 against 1.55 on 18^3, p = 7 2.15 against 2.16 on
// 12^3; SF-KG, whose pairs cost less, 14% more at p = 1 down to 4% at p = 7.
template <int N, int VF, bool XF, int EPB>
__device__ __noinline__ void out_of_range(double* smem, const double* q, double* dqdt, const double* geom,
                                          const double* jinv, const int32_t* nbr, double* trace, int64_t K,
                                          const Ops& ops, const Phys& ph, const double* qext, const double* src,
                                          const double* nsurf, const double* fnorm) {
    element_f64<N, VF, XF, EPB>(smem, q, dqdt, geom, jinv, nbr, trace, K, ops, ph, qext, src, nsurf, fnorm);
}

// Euler flux contracted with n, from density, velocity, pressure and specific enthalpy
__device__ __forceinline__ void euler_flux(double rho, double u0, double u1, double u2, double p, double H, double n0,
                                           double n1, double n2, double (&f)[5]) {
    f[0] = rho * fma(u2, n2, fma(u1, n1, u0 * n0));
    f[1] = fma(f[0], u0, p * n0);
    f[2] = fma(f[0], u1, p * n1);
    f[3] = fma(f[0], u2, p * n2);
    f[4] = f[0] * H;
}

// The two-point flux in fixed point (units 2^k0, 2^km, 2^k5), contracted with n.
template <int VF>
__device__ __forceinline__ void two_point(const PrimFx& a, const PrimFx& b, Fx n0, Fx n1, Fx n2, Fx cg, double inv_gm1,
                                          const FixScale& s, long long (&f)[5]) {
    if constexpr (VF == kFluxESC) {
        ec_flux_fx(a, b, n0, n1, n2, cg, s, LogMeanF64{a.r, b.r, a.b, b.b, s, inv_gm1}, f);
    } else {
        kg_flux_fx(a, b, n0, n1, n2, s, f);
    }
}

// out_i = sum_j M_ij in_j along one line of N Q60 values
template <int N>
__device__ __forceinline__ void line_product(const Fx (&v)[N], const Fx (&M)[kMaxN][kMaxN], long long (&out)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        long long h = 0, m = kFxHalf + N * kFxLow;
#pragma unroll
        for (int j = 0; j < N; ++j) fx_mac(h, m, M[i][j], v[j]);
        out[i] = h + (m >> 30);
    }
}

// XF: the kernel also handles the matrix dissipation, the interior penalty, boundary faces with an
// exterior state, a source term and surface metrics (compiled only into the instantiations of contexts
// that use them)
template <int N, int VF, bool XF, bool WIDE>
__global__ void __launch_bounds__(FixCfg<N, VF, WIDE>::THREADS, FixCfg<N, VF, WIDE>::MINB)
rhs_fix_f64(const double* __restrict__ q, double* __restrict__ dqdt, const double* __restrict__ geom,
            const double* __restrict__ jinv, const int32_t* __restrict__ nbr, double* __restrict__ trace, int64_t K,
            const __grid_constant__ Ops ops, const __grid_constant__ Phys ph, const double* __restrict__ qext,
            const double* __restrict__ src, const double* __restrict__ nsurf, const double* __restrict__ fnorm,
            const int32_t* __restrict__ kn) {
    using C = FixCfg<N, VF, WIDE>;
    constexpr int N2 = C::N2, N3 = C::N3, EPB = C::EPB, SL = C::SL, NP = C::NP, NE = VF == kFluxKG ? 12 : 10;
    extern __shared__ double smem[];
    __shared__ int sE[EPB][NE];                  // largest exponents (of 4096 - E for the smallest)
    __shared__ FixScale sScale[EPB];
    __shared__ unsigned sMag[EPB][2];            // magnitude bits of theta: w2..w4, w5
    __shared__ Fx sS[(N / 2) * N];
    __shared__ double sW[N];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int el_loc = t / N3;
    const int node = t - el_loc * N3;
    const int64_t el = (int64_t)blockIdx.x * EPB + el_loc;
    const bool active = el_loc < EPB && el < K;
    const int n_el = (int)(K - (int64_t)blockIdx.x * EPB < EPB ? K - (int64_t)blockIdx.x * EPB : EPB);
    const int i1 = node % N, i2 = (node / N) % N, i3 = node / N2;
    double* sm = smem + (size_t)el_loc * C::SM;
    Fx* X = reinterpret_cast<Fx*>(sm);
    const int own_slot = slot<N>(i1, i2, i3);
    const int64_t eoff = el * 5 * N3;
    for (int i = t; i < EPB * NE; i += C::THREADS)
        sE[i / NE][i % NE] = i % NE == 5 && i / NE < n_el ? kn[(int64_t)blockIdx.x * EPB + i / NE] : 0;
    if (t < EPB) sMag[t][0] = sMag[t][1] = 0;
    for (int i = t; i < (N / 2) * N; i += C::THREADS) sS[i] = ops.SF[i / N][i % N];
    for (int i = t; i < N; i += C::THREADS) sW[i] = ops.winv[i];
    __syncthreads();

    // ---- 0. primitives, exponents, scaling
    double Jinv = 0.0, Y = 0.0, Z = 0.0;
    if (active) {
        double qv[5], RT, pi[NP];
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = q[eoff + v * N3 + node];
        Jinv = jinv[el * N3 + node];
        int E[NE];
        E[5] = 0;
#pragma unroll
        for (int c = 0; c < 9; ++c) sm[C::XN + c * SL + own_slot] = geom[(el * 10 + 1 + c) * N3 + node];
        pair_inputs<VF>(qv, ph, pi, RT);
#pragma unroll
        for (int i = 0; i < NP; ++i) sm[C::XP + i * SL + own_slot] = pi[i];
        sm[C::P + node] = RT;
        rhs_exponents(pi, E);
        Y = ph.mu * RT * Jinv;                   // velocity gradient to stress
        Z = ph.kappa_R * RT * RT * Jinv;         // dw5 to heat flux
        E[6] = biased_exp(Y);
        E[7] = biased_exp(Z);
        block_max<EPB == 1 || N3 % 32 == 0>(sE[el_loc], el_loc, E, lane);
    }
#pragma unroll 1
    for (int id = t; id < n_el * 6 * N2; id += C::THREADS) {
        const int e = id / (6 * N2), fn = id - e * 6 * N2;
        const int64_t ee = (int64_t)blockIdx.x * EPB + e;
        const int l = fn / (2 * N2);
        const int rem = fn - l * 2 * N2;
        const int side = rem / N2, fi = rem - side * N2;
        const int st = dir_stride<N>(l);
        const int base = line_base<N>(l, fi % N, fi / N);
        const int64_t nb = nbr[ee * 6 + 2 * l + side];
        const double* qn = q + nb * 5 * N3 + base + (side ? 0 : (N - 1) * st);
        int E[NE];
        E[5] = E[6] = E[7] = 0;
        // a boundary face (neighbour -1, bounded boxes only) sees the exterior state at its own nodes
        if constexpr (XF) {
            if (nb < 0) qn = qext + ee * 5 * N3 + base + (side ? (N - 1) * st : 0);
        }
        double qv[5], RT, pi[NP];
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = qn[v * N3];
        pair_inputs<VF>(qv, ph, pi, RT);
        double* f = smem + (size_t)e * C::SM + C::F + fn;
#pragma unroll
        for (int i = 0; i < NP; ++i) f[i * 6 * N2] = pi[i];
        f[NP * 6 * N2] = sqrt_newton(ph.gamma * RT);
        rhs_exponents(pi, E);
        block_max<EPB == 1 || (6 * N2) % 32 == 0>(sE[e], e, E, lane);
    }
    __syncthreads();
    bool ok;
    if constexpr (EPB <= 2) ok = rhs_range_ok(sE[0]) && (n_el < 2 || rhs_range_ok(sE[EPB - 1]));
    else ok = __syncthreads_and(t >= n_el || rhs_range_ok(sE[t]));
    if (!ok) {
        __syncthreads();
        out_of_range<N, VF, XF, EPB>(smem, q, dqdt, geom, jinv, nbr, trace, K, ops, ph, qext, src, nsurf, fnorm);
        return;
    }
    if (active) {
        const FixScale s = element_scale<VF>(sE[el_loc], ops.kg);
        if (node == 0) sScale[el_loc] = s;
        if constexpr (VF == kFluxDC) {
            // nodal contravariant fluxes Ftilde_l
            const double* pi = sm + C::XP + own_slot;
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                const double* n = sm + C::XN + 3 * l * SL + own_slot;
                double f[5];
                euler_flux(2.0 * pi[0], 2.0 * pi[SL], 2.0 * pi[2 * SL], 2.0 * pi[3 * SL], 2.0 * pi[6 * SL], pi[5 * SL], n[0], n[SL],
                           n[2 * SL], f);
#pragma unroll
                for (int v = 0; v < 5; ++v) sm[C::R + (5 * l + v) * SL + own_slot] = f[v];
            }
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            const int i = C::XN + c * SL + own_slot;
            X[i] = fx_split(fx_from_double(sm[i], s.kn));
        }
        Fx* XP = X + C::XP + own_slot;
        scale_inputs<VF>(sm + C::XP + own_slot, XP, SL, s);
#pragma unroll
        for (int m = 0; m < 3; ++m)              // w = 2 beta u in units 2^(kb + ku)
            X[C::XW + m * SL + own_slot] = fx_split(fx_mul(XP[4 * SL], XP[(1 + m) * SL]) * 4);
    }
#pragma unroll 1
    for (int id = t; id < n_el * 6 * N2; id += C::THREADS) {
        const int e = id / (6 * N2), fn = id - e * 6 * N2;
        double* f = smem + (size_t)e * C::SM + C::F + fn;
        scale_inputs<VF>(f, reinterpret_cast<Fx*>(f), 6 * N2, element_scale<VF>(sE[e], ops.kg));
    }
    __syncthreads();

    // ---- 1. volume flux differencing
    if constexpr (VF == kFluxDC) {
        // the nodal fluxes' differences along the lines, sum_j S_ij (F_i + F_j) with the own flux left out, which at
        // the end nodes is half the interface flux's own part; in fixed point under the line's largest exponent, in
        // place
#pragma unroll 1
        for (int id = t; id < n_el * 15 * N2; id += C::THREADS) {
            const int e = id / (15 * N2), r = id - e * 15 * N2;
            const int lv = r / N2, li = r - lv * N2;
            const int l = lv / 5, c1 = li % N, c2 = li / N;
            double* R = smem + (size_t)e * C::SM + C::R + lv * SL;
            double f[N];
            int k = 0;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                f[j] = R[line_slot<N>(l, j, c1, c2)];
                k = max(k, biased_exp(f[j]));
            }
            k -= 1021;
            Fx x[N];
            long long out[N];
#pragma unroll
            for (int j = 0; j < N; ++j) x[j] = fx_split(fx_from_double(f[j], k));
            line_product<N>(x, ops.MF, out);
#pragma unroll
            for (int j = 0; j < N; ++j) R[line_slot<N>(l, j, c1, c2)] = -ops.winv[j] * fx_to_double(out[j], k);
        }
    } else {
        const int lw = lane / N, i = lane - lw * N;
#pragma unroll 1
        for (int task = warp; task < 3 * C::TPD; task += C::WARPS) {
            const int l = task / C::TPD;
            int line = (task - l * C::TPD) * C::LPW + lw;
            const bool go = lw < C::LPW && line < n_el * N2;
            line = go ? line : 0;
            const int e = line / N2, li = line - e * N2;
            const int c1 = li % N, c2 = li / N;
            double* se = smem + (size_t)e * C::SM;
            const Fx* XP = reinterpret_cast<const Fx*>(se) + C::XP;
            const Fx* XN = reinterpret_cast<const Fx*>(se) + C::XN + 3 * l * SL;
            const FixScale& s = sScale[e];
            const int ii = line_slot<N>(l, i < N ? i : 0, c1, c2);
            const PrimFx a = load_inputs<VF>(XP + ii, SL);
            const Fx na0 = XN[ii], na1 = XN[SL + ii], na2 = XN[2 * SL + ii];
            unsigned long long acc[5] = {0, 0, 0, 0, 0};
#pragma unroll 1
            for (int k = 1; k <= N / 2; ++k) {
                const int j = i + k < N ? i + k : i + k - N;
                long long Pv[5] = {0, 0, 0, 0, 0};
                if (go && (2 * k < N || i < k)) {
                    const int jj = line_slot<N>(l, j, c1, c2);
                    const PrimFx b = load_inputs<VF>(XP + jj, SL);
                    // the flux is linear in n: contracted with S_ij (n_i + n_j), twice the averaged metric
                    // times half the pair coefficient
                    const Fx S = sS[(k - 1) * N + i];
                    const Fx n0 = fx_split(fx_mul<2>(S, fx_add(na0, XN[jj]))), n1 = fx_split(fx_mul<2>(S, fx_add(na1, XN[SL + jj]))),
                             n2 = fx_split(fx_mul<2>(S, fx_add(na2, XN[2 * SL + jj])));
                    two_point<VF>(a, b, n0, n1, n2, ops.CG, ph.inv_gm1, s, Pv);
#pragma unroll
                    for (int v = 0; v < 5; ++v) acc[v] -= (unsigned long long)Pv[v];
                }
                const int from = (lw * N + (i >= k ? i - k : i - k + N)) & 31;
#pragma unroll
                for (int v = 0; v < 5; ++v) acc[v] += (unsigned long long)__shfl_sync(0xffffffffu, Pv[v], from);
            }
            if (go) {
                double* R = se + C::R + l * 5 * SL + ii;
                const double w = sW[i];
#pragma unroll
                for (int v = 0; v < 5; ++v)
                    R[v * SL] = w * fx_to_double((long long)acc[v], v == 0 ? s.k0 : (v == 4 ? s.k5 : s.km));
            }
        }
    }
    __syncthreads();

    // ---- 2. interface SAT: -(E_ii f_EC(own, nbr).n_J + lambda/2 (q_own - q_nbr)) / w_i, into the
    // direction's result
#pragma unroll 1
    for (int id = t; id < n_el * 6 * N2; id += C::THREADS) {
        const int e = id / (6 * N2), fn = id - e * 6 * N2;
        const int64_t ee = (int64_t)blockIdx.x * EPB + e;
        double* se = smem + (size_t)e * C::SM;
        const Fx* Xe = reinterpret_cast<const Fx*>(se);
        const FixScale& s = sScale[e];
        const int l = fn / (2 * N2);
        const int rem = fn - l * 2 * N2;
        const int side = rem / N2, fi = rem - side * N2;
        const int st = dir_stride<N>(l);
        const int base = line_base<N>(l, fi % N, fi / N);
        const int own = base + (side ? (N - 1) * st : 0);
        const int os = line_slot<N>(l, side ? N - 1 : 0, fi % N, fi / N);
        const int64_t nb = nbr[ee * 6 + 2 * l + side];
        const double* qn = q + nb * 5 * N3 + base + (side ? 0 : (N - 1) * st);
        bool bnd = false;
        if constexpr (XF) {
            bnd = nb < 0;
            if (bnd) qn = qext + ee * 5 * N3 + own;
        }
        const Fx* XP = Xe + C::XP + os;
        const Fx* g = Xe + C::F + fn;
        const PrimFx a = load_inputs<VF>(XP, SL), b = load_inputs<VF>(g, 6 * N2);
        Fx n0 = Xe[C::XN + 3 * l * SL + os], n1 = Xe[C::XN + (3 * l + 1) * SL + os], n2 = Xe[C::XN + (3 * l + 2) * SL + os];
        [[maybe_unused]] double nd[3];
        if constexpr (XF) {
            // optimized metrics: the interface terms take the analytic surface metrics (the own
            // flux, cancelled against the volume term's boundary part, keeps the volume metrics)
            const double* ns = nsurf ? nsurf + (ee * 6 + 2 * l + side) * 3 * N2 + fi : geom + (ee * 10 + 1 + 3 * l) * N3 + own;
            const int sn = nsurf ? N2 : N3;
            nd[0] = ns[0];
            nd[1] = ns[sn];
            nd[2] = ns[2 * sn];
            if (nsurf) {
                n0 = fx_split(fx_from_double(nd[0], s.kn));
                n1 = fx_split(fx_from_double(nd[1], s.kn));
                n2 = fx_split(fx_from_double(nd[2], s.kn));
            }
        }
        [[maybe_unused]] long long f[5];
        [[maybe_unused]] double fnb[5];          // DC: the neighbour's nodal flux
        if constexpr (VF == kFluxDC) {
            const double* gd = se + C::F + fn;
            if constexpr (!XF) {
                const double* ns = geom + (ee * 10 + 1 + 3 * l) * N3 + own;
                nd[0] = ns[0];
                nd[1] = ns[N3];
                nd[2] = ns[2 * N3];
            }
            const double ri = rcp_cubic(qn[0]);
            euler_flux(qn[0], qn[N3] * ri, qn[2 * N3] * ri, qn[3 * N3] * ri, 2.0 * gd[6 * 6 * N2], gd[5 * 6 * N2], nd[0], nd[1],
                       nd[2], fnb);
            if constexpr (XF) {
                // optimized metrics: the own flux left out of the volume term was one with the volume metrics
                if (nsurf) {
                    const double *qo = q + ee * 5 * N3 + own, *nv = geom + (ee * 10 + 1 + 3 * l) * N3 + own;
                    const double ro = rcp_cubic(qo[0]), RT = se[C::P + own];
                    const double u0 = qo[N3] * ro, u1 = qo[2 * N3] * ro, u2 = qo[3 * N3] * ro;
                    double fo[5];
                    euler_flux(qo[0], u0, u1, u2, qo[0] * RT, fma(ph.gamma * ph.inv_gm1, RT, 0.5 * fma(u2, u2, fma(u1, u1, u0 * u0))),
                               nd[0] - nv[0], nd[1] - nv[N3], nd[2] - nv[2 * N3], fo);
#pragma unroll
                    for (int v = 0; v < 5; ++v) fnb[v] += fo[v];
                }
            }
        } else {
            two_point<VF>(a, b, n0, n1, n2, ops.CG, ph.inv_gm1, s, f);
        }
        double lam = 0.0;
        double dm[5] = {0.0, 0.0, 0.0, 0.0, 0.0};      // 1/2 D (w_own - w_nbr) + interior penalty
        if (XF && (ph.dissipation == 2 || ph.ip_coef > 0.0)) {
            double qv[5], jw[5], r[5], RTo, RTn, co, cn;
            Prim so, sn;
            FaceAvg fa;
#pragma unroll
            for (int v = 0; v < 5; ++v) qv[v] = q[ee * 5 * N3 + v * N3 + own];
            to_prim(qv, ph, so, RTo, co);
#pragma unroll
            for (int v = 0; v < 5; ++v) qv[v] = qn[v * N3];
            to_prim(qv, ph, sn, RTn, cn);
            face_jump_avg(so, RTo, sn, RTn, ph, jw, r, fa);
            if (ph.dissipation == 2) {
                matrix_dissipation(fa, jw, r, nd[0], nd[1], nd[2], ph, dm);
#pragma unroll
                for (int v = 0; v < 5; ++v) dm[v] *= 0.5;
            }
            if (ph.ip_coef > 0.0) {
                // sigma mu |n_J| / h with h = (J_own + J_nbr)/|n_J|
                const double nsq = nd[0] * nd[0] + nd[1] * nd[1] + nd[2] * nd[2];
                const double Jo = geom[ee * 10 * N3 + own];
                const double Jn = bnd ? Jo : geom[nb * 10 * N3 + base + (side ? 0 : (N - 1) * st)];
                const double cip = ph.ip_coef * ph.mu * nsq / (Jo + Jn);
#pragma unroll
                for (int v = 0; v < 5; ++v) dm[v] = fma(cip, r[v], dm[v]);
            }
        }
        if (ph.dissipation == 1) {
            // |u.n| of both sides in Q60, c |n_J| in float64
            const double nn = fnorm[(ee * 6 + 2 * l + side) * N2 + fi];
            const double co = sqrt_newton(ph.gamma * se[C::P + own]), cn = se[C::F + NP * 6 * N2 + fn];
            const double uo = fx_to_double(fx_dot(a.u0, n0, a.u1, n1, a.u2, n2), s.ku + s.kn + 1);
            const double un = fx_to_double(fx_dot(b.u0, n0, b.u1, n1, b.u2, n2), s.ku + s.kn + 1);
            lam = ops.winv[0] * (0.5 * fmax(fma(co, nn, fabs(uo)), fma(cn, nn, fabs(un))));
        }
        const double wi = side ? -ops.winv[N - 1] : ops.winv[0];
        double* R = se + C::R + l * 5 * SL + os;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double r;
            if constexpr (VF == kFluxDC) r = fma(0.5 * wi, fnb[v], R[v * SL]);
            else r = fma(wi, fx_to_double(f[v], v == 0 ? s.k0 : (v == 4 ? s.k5 : s.km)), R[v * SL]);
            if (ph.dissipation == 1) r = fma(-lam, q[ee * 5 * N3 + v * N3 + own] - qn[v * N3], r);
            if constexpr (XF) r = fma(-ops.winv[0], dm[v], r);
            R[v * SL] = r;
        }
    }
    __syncthreads();
    double res[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (active) {
        const double* R = sm + C::R + own_slot;
#pragma unroll
        for (int v = 0; v < 5; ++v) res[v] = R[v * SL] + R[(5 + v) * SL] + R[(10 + v) * SL];
    }

    // ---- 3. viscous terms
    if (ph.viscous) {
        __syncthreads();                         // the results' space becomes theta's
        // theta_a[k] = D_a w_k + lift: w2..w4 (k < 3), beta for w5 = -2 beta (k = 3)
#pragma unroll 1
        for (int id = t; id < n_el * 12 * N2; id += C::THREADS) {
            const int e = id / (12 * N2), r = id - e * 12 * N2;
            const int lk = r / N2, li = r - lk * N2;
            const int l = lk >> 2, k = lk & 3;
            const int c1 = li % N, c2 = li / N;
            Fx* Xe = reinterpret_cast<Fx*>(smem + (size_t)e * C::SM);
            const Fx* W = Xe + (k < 3 ? C::XW + k * SL : C::XP + 4 * SL);
            Fx v[N];
            long long out[N];
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = W[line_slot<N>(l, j, c1, c2)];
            long long lift[2];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const Fx* g = Xe + C::F + (2 * l + side) * N2 + li;
                Fx wn = g[24 * N2];
                if (k < 3) wn = fx_split(fx_mul(wn, g[(1 + k) * 6 * N2]) * 4);
                const Fx wo = v[side ? N - 1 : 0];
                lift[side] = fx_mul<0>(ops.LF, side ? fx_sub(wn, wo) : fx_sub(wo, wn));
            }
            line_product<N>(v, ops.DF, out);     // in units 2^kD
            out[0] += lift[0];
            out[N - 1] += lift[1];
            long long* T = reinterpret_cast<long long*>(Xe + C::R + lk * SL);
            unsigned mag = 0;                    // bits of the magnitudes, units of 2^-31
#pragma unroll
            for (int j = 0; j < N; ++j) {
                T[line_slot<N>(l, j, c1, c2)] = out[j];
                mag |= (unsigned)((out[j] ^ (out[j] >> 63)) >> 29);
            }
            if constexpr (N2 % 32 == 0) {        // one variable and element per warp
                mag = __reduce_or_sync(0xffffffffu, mag);
                if (lane == 0) atomicOr(&sMag[e][k == 3], mag);
            } else {
                atomicOr(&sMag[e][k == 3], mag);
            }
        }
        __syncthreads();
        if (active) {
            // theta shifted up to the element's largest: its derivatives of nearly constant fields use few
            // of their bits, and what follows would round them away
            const int sw = max(__clz(sMag[el_loc][0]) - 1, 0), sb = max(__clz(sMag[el_loc][1]) - 1, 0);
            const ViscScale s = visc_scale(sScale[el_loc], sw, sb, ops.kD);
            const long long* T = reinterpret_cast<const long long*>(X + C::R + own_slot);
            Fx* XN = X + C::XN + own_slot;
            Fx* XP = X + C::XP + own_slot;
            // A[k][m] = sum_a Ja_am theta_a[k] + u_k (the same of w5): du_k/dx_m without its factor J^-1 RT
            long long A[3][3];
            Fx Gb[3];
#pragma unroll
            for (int m = 0; m < 3; ++m)
                Gb[m] = fx_split(fx_dot(XN[m * SL], fx_split(T[3 * SL] << sb), XN[(3 + m) * SL], fx_split(T[7 * SL] << sb),
                                        XN[(6 + m) * SL], fx_split(T[11 * SL] << sb)));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Fx t0 = fx_split(T[k * SL] << sw), t1 = fx_split(T[(4 + k) * SL] << sw), t2 = fx_split(T[(8 + k) * SL] << sw);
                const Fx u = XP[(1 + k) * SL];
#pragma unroll
                for (int m = 0; m < 3; ++m)
                    A[k][m] = (fx_dot(XN[m * SL], t0, XN[(3 + m) * SL], t1, XN[(6 + m) * SL], t2) >> s.sg) - (fx_mul(u, Gb[m]) >> s.su);
            }
            const Fx y = fx_split(fx_from_double(Y, s.ky)), z = fx_split(fx_from_double(Z, s.kz));
            const long long tr = fx_mul(fx_split((A[0][0] + A[1][1] + A[2][2] + 2) >> 2), Fx{715827882, 715827883});
            // stress mu (du_i/dx_m + du_m/dx_i - 2/3 div): xx, yy, zz, yz, xz, xy
            Fx tau[6];
#pragma unroll
            for (int m = 0; m < 3; ++m) tau[m] = fx_split(fx_mul(y, fx_split(((A[m][m] + 1) >> 1) - tr)));
            tau[3] = fx_split(fx_mul(y, fx_split((A[1][2] + A[2][1] + 2) >> 2)));
            tau[4] = fx_split(fx_mul(y, fx_split((A[0][2] + A[2][0] + 2) >> 2)));
            tau[5] = fx_split(fx_mul(y, fx_split((A[0][1] + A[1][0] + 2) >> 2)));
            // energy flux tau u + heat flux
            Fx en[3];
            {
                const Fx u0 = XP[SL], u1 = XP[2 * SL], u2 = XP[3 * SL];
                const long long e0 = fx_dot(tau[0], u0, tau[5], u1, tau[4], u2);
                const long long e1 = fx_dot(tau[5], u0, tau[1], u1, tau[3], u2);
                const long long e2 = fx_dot(tau[4], u0, tau[3], u1, tau[2], u2);
                en[0] = fx_split(((e0 + s.he) >> s.se) - ((fx_mul(z, Gb[0]) + s.hz) >> s.sz));
                en[1] = fx_split(((e1 + s.he) >> s.se) - ((fx_mul(z, Gb[1]) + s.hz) >> s.sz));
                en[2] = fx_split(((e2 + s.he) >> s.se) - ((fx_mul(z, Gb[2]) + s.hz) >> s.sz));
            }
            // contravariant fluxes Ftilde_l, each over the metric row it used and an unused primitive
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                const Fx n0 = XN[3 * l * SL], n1 = XN[(3 * l + 1) * SL], n2 = XN[(3 * l + 2) * SL];
                long long Ft[4];
                Ft[0] = fx_dot(n0, tau[0], n1, tau[5], n2, tau[4]);
                Ft[1] = fx_dot(n0, tau[5], n1, tau[1], n2, tau[3]);
                Ft[2] = fx_dot(n0, tau[4], n1, tau[3], n2, tau[2]);
                Ft[3] = fx_dot(n0, en[0], n1, en[1], n2, en[2]);
#pragma unroll
                for (int k = 0; k < 3; ++k) XN[(3 * l + k) * SL] = fx_split(Ft[k]);
                XP[l * SL] = fx_split(Ft[3]);
                const int il = l == 0 ? i1 : (l == 1 ? i2 : i3);
                if (il == 0 || il == N - 1) {
                    const int side = il == N - 1;
                    const int fi = l == 0 ? (i2 + N * i3) : (l == 1 ? (i1 + N * i3) : (i1 + N * i2));
                    double* tr_out = trace + ((el * 6 + 2 * l + side) * 4) * N2 + fi;
#pragma unroll
                    for (int k = 0; k < 4; ++k) tr_out[k * N2] = fx_to_double(Ft[k], k < 3 ? s.kf : s.kh);
                }
            }
        }
        __syncthreads();
        // the fluxes' derivatives along their own direction, in place
#pragma unroll 1
        for (int id = t; id < n_el * 12 * N2; id += C::THREADS) {
            const int e = id / (12 * N2), r = id - e * 12 * N2;
            const int lk = r / N2, li = r - lk * N2;
            const int l = lk >> 2, k = lk & 3;
            const int c1 = li % N, c2 = li / N;
            Fx* W = reinterpret_cast<Fx*>(smem + (size_t)e * C::SM) + (k < 3 ? C::XN + (3 * l + k) * SL : C::XP + l * SL);
            Fx v[N];
            long long out[N];
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = W[line_slot<N>(l, j, c1, c2)];
            line_product<N>(v, ops.DF, out);
            long long* D = reinterpret_cast<long long*>(W);
#pragma unroll
            for (int j = 0; j < N; ++j) D[line_slot<N>(l, j, c1, c2)] = out[j];
        }
        __syncthreads();
        if (active) {
            const int sw = max(__clz(sMag[el_loc][0]) - 1, 0), sb = max(__clz(sMag[el_loc][1]) - 1, 0);
            const ViscScale s = visc_scale(sScale[el_loc], sw, sb, ops.kD);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long* D = reinterpret_cast<const long long*>(X + (k < 3 ? C::XN + k * SL : C::XP) + own_slot);
                const int st = k < 3 ? 3 * SL : SL;
                res[1 + k] += fx_to_double(D[0] + D[st] + D[2 * st], (k < 3 ? s.kf : s.kh) + ops.kD);
            }
        }
    }
    if (active) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double r = res[v] * Jinv;
            if constexpr (XF) {
                if (src) r = fma(res[v], Jinv, src[eoff + v * N3 + node]);
            }
            dqdt[eoff + v * N3 + node] = r;
        }
    }
}

// the float64 form runs in the same shared memory
template <int N, int VF, bool WIDE>
constexpr size_t fix_smem() {
    constexpr int sm = FixCfg<N, VF, WIDE>::SM > Cfg<N>::SM ? FixCfg<N, VF, WIDE>::SM : Cfg<N>::SM;
    return (size_t)FixCfg<N, VF, WIDE>::EPB * sm * sizeof(double);
}

template <int N, int VF, bool XF, bool WIDE>
cudaError_t launch_w(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    using C = FixCfg<N, VF, WIDE>;
    const unsigned grid = (unsigned)((c->K + C::EPB - 1) / C::EPB);
    rhs_fix_f64<N, VF, XF, WIDE><<<grid, C::THREADS, fix_smem<N, VF, WIDE>(), s>>>(
        q, dqdt, c->d_geom, c->d_jinv, c->d_nbr, (double*)c->d_trace, c->K, c->ops, c->phys, c->d_qext, c->d_src,
        c->d_nsurf, c->d_fnorm, c->d_kn);
    return cudaGetLastError();
}

// the float64 form as a kernel of its own, for meshes of stretched elements
template <int N, int VF, bool XF>
__global__ void __launch_bounds__(Cfg<N>::THREADS, Cfg<N>::MINB)
rhs_f64(const double* __restrict__ q, double* __restrict__ dqdt, const double* __restrict__ geom,
        const double* __restrict__ jinv, const int32_t* __restrict__ nbr, double* __restrict__ trace, int64_t K,
        const __grid_constant__ Ops ops, const __grid_constant__ Phys ph, const double* __restrict__ qext,
        const double* __restrict__ src, const double* __restrict__ nsurf, const double* __restrict__ fnorm) {
    extern __shared__ double smem[];
    element_f64<N, VF, XF>(smem, q, dqdt, geom, jinv, nbr, trace, K, ops, ph, qext, src, nsurf, fnorm);
}

template <int N, int VF, bool XF>
cudaError_t launch_f64(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    using C = Cfg<N>;
    const unsigned grid = (unsigned)((c->K + C::EPB - 1) / C::EPB);
    rhs_f64<N, VF, XF><<<grid, C::THREADS, C::EPB * C::SM * sizeof(double), s>>>(
        q, dqdt, c->d_geom, c->d_jinv, c->d_nbr, (double*)c->d_trace, c->K, c->ops, c->phys, c->d_qext, c->d_src,
        c->d_nsurf, c->d_fnorm);
    return cudaGetLastError();
}

// Elements per SM up to which the wide form is taken (0: never), per residual with its face kernel, normal
// against wide form: N = 2 512 elements 36.0 -> 20.7 us, N = 3 512 32.9 -> 24.7, N = 4 64 30 -> 20, 216
// 30.9 -> 24.7, 343 37.0 -> 35.0, 512 37.1 -> 39.1, N = 5 125 35.0 -> 26.8, 216 41.1 -> 41.8, N = 7 125
// 53.4 -> 47.3, 343 121.5 -> 125.1; N = 6 and 8 gain nothing (37.0 and 63.6 us for up to one element per SM).
// The instances with the optional interface terms keep fewer CTAs resident, so their line lies lower (bounded box,
// normal against wide: N = 2 576 elements ES-C 0.89 of the time, 720 1.10, 900 1.16, DC 0.84, 1.09, 1.14, SF-KG 900
// 39.1 -> 32.9 us; N = 3 448 elements 0.7, 576 1.06 to 1.11; N = 4 294 DC 31.9 -> 39.1 us, the others 0.8).
constexpr int wide_upto(int n, int vf, bool xf) {
    return n == 2 ? (xf && vf != kFluxKG ? 4 : 6)
                  : (n == 3 ? (xf ? 3 : 4) : (n == 4 ? (xf && vf == kFluxDC ? 1 : 2) : (n == 5 || n == 7 ? 1 : 0)));
}

template <int N, int VF, bool XF>
cudaError_t launch_n(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    if (c->float64_form) return launch_f64<N, VF, XF>(c, q, dqdt, s);
    if constexpr (wide_upto(N, VF, XF) > 0)
        if (c->K <= (int64_t)wide_upto(N, VF, XF) * sm_count()) return launch_w<N, VF, XF, true>(c, q, dqdt, s);
    return launch_w<N, VF, XF, false>(c, q, dqdt, s);
}

template <int N, int VF, bool XF>
cudaError_t prepare_n(const esdc_ctx* c) {
    constexpr cudaFuncAttribute kAttr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (c->float64_form) return cudaFuncSetAttribute(rhs_f64<N, VF, XF>, kAttr, (int)(Cfg<N>::EPB * Cfg<N>::SM * sizeof(double)));
    const cudaError_t e = cudaFuncSetAttribute(rhs_fix_f64<N, VF, XF, false>, kAttr, (int)fix_smem<N, VF, false>());
    if constexpr (wide_upto(N, VF, XF) > 0)
        if (e == cudaSuccess) return cudaFuncSetAttribute(rhs_fix_f64<N, VF, XF, true>, kAttr, (int)fix_smem<N, VF, true>());
    return e;
}

template <int VF, bool XF>
cudaError_t prepare_vf(const esdc_ctx* c) {
    switch (c->N) {
        case 2: return prepare_n<2, VF, XF>(c);
        case 3: return prepare_n<3, VF, XF>(c);
        case 4: return prepare_n<4, VF, XF>(c);
        case 5: return prepare_n<5, VF, XF>(c);
        case 6: return prepare_n<6, VF, XF>(c);
        case 7: return prepare_n<7, VF, XF>(c);
        case 8: return prepare_n<8, VF, XF>(c);
        default: return cudaErrorInvalidValue;
    }
}

template <int VF, bool XF>
cudaError_t launch_vf(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    switch (c->N) {
        case 2: return launch_n<2, VF, XF>(c, q, dqdt, s);
        case 3: return launch_n<3, VF, XF>(c, q, dqdt, s);
        case 4: return launch_n<4, VF, XF>(c, q, dqdt, s);
        case 5: return launch_n<5, VF, XF>(c, q, dqdt, s);
        case 6: return launch_n<6, VF, XF>(c, q, dqdt, s);
        case 7: return launch_n<7, VF, XF>(c, q, dqdt, s);
        case 8: return launch_n<8, VF, XF>(c, q, dqdt, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace esdc
