// Volume part of the ES-C adjoint in block fixed point (fix_f64.cuh): the pair cotangents
// mu = 2 S_ij (lt_j/w_j - lt_i/w_i), lt = lambda/J, pulled back through the two-point flux to both nodes,
// summed per node over the three directions and mapped to the conserved variables, where adjoint_f64.cu starts
// from.
//
// The float64 reverse takes ~105 operations of 64 clocks per warp and scheduler a pair; here a pair takes
// about fifty 60-bit products of 17.  Same mapping as the residual's pair loop (rhs_fix.cuh): one thread per
// (node, direction), whole lines side by side in a warp, pair (i, i + k mod N) at cyclic distance k; the
// partner's lambda/(J w) and the results for it travel by shuffle.  The flux is linear in the metric, so
// S_ij multiplies n_i + n_j and the cotangent is the plain difference of lambda/(J w).  Results are linear in
// lambda, which may vary by orders within an element (quadrature weights alone by (w_mid/w_end)^2, 130 at p = 7):
// each line takes it under its own largest value and shifts its sums back.  Elements outside the fixed-point range
// (primitives as in the residual, or lambda/J beyond it) take the float64 reverse.
#include <cuda_runtime.h>

#include "adj_pair_f64.cuh"
#include "esdc_internal.h"
#include "fix_f64.cuh"
#include "kernels.h"
#include "rhs_fix.cuh"

namespace esdc {
namespace {

template <int N>
struct AdjCfg {
    static constexpr int N2 = N * N, N3 = N * N * N, SL = FixSlot<N>::SL;
    static constexpr int EPB = Cfg<N>::EPB;
    static constexpr int THREADS = (EPB * N3 + 31) / 32 * 32, WARPS = THREADS / 32;
    static constexpr int LPW = 32 / N, TPD = (EPB * N2 + LPW - 1) / LPW;
    // shared memory per element in 8-byte units: metric rows 9 | pair inputs 6 | lambda/J 5 | results 3 x 6
    static constexpr int XN = 0, XP = 9 * SL, LT = 15 * SL, B = 20 * SL, SM = 38 * SL;
    static constexpr int MINB = N == 8 ? 1 : (N >= 6 ? 2 : 4);
};

// Logarithmic means and their derivatives beyond the series, in float64 from the fixed-point inputs.
__device__ __noinline__ void rho_mean_f64(long long a, long long b, int k, LogMeansFx& m) {
    const double x = 2.0 * fx_to_double(a, k), y = 2.0 * fx_to_double(b, k), d = x - y, l = log(x / y), L = d / l;
    m.rl = fx_from_double(L, k);
    m.La = fx_from_double((1.0 - L / x) / l, 0);
    m.Lb = fx_from_double((L / y - 1.0) / l, 0);
}
__device__ __noinline__ void beta_mean_f64(long long a, long long b, int k, double hig, int kA, int kd, LogMeansFx& m) {
    const double x = fx_to_double(a, k), y = fx_to_double(b, k), d = x - y, I = log(x / y) / d;
    m.A = fx_from_double(hig * I, kA);
    m.DA = fx_from_double(hig * (1.0 / x - I) / d, kd);
    m.DB = fx_from_double(hig * (I - 1.0 / y) / d, kd);
}
struct AdjMeansF64 {
    Fx ra, rb, ba, bb;
    const FixScale& s;
    int kd;
    double hig;
    __device__ __forceinline__ void rho(LogMeansFx& m) const { rho_mean_f64(fx_join(ra), fx_join(rb), s.kr, m); }
    __device__ __forceinline__ void beta(LogMeansFx& m) const {
        beta_mean_f64(fx_join(ba), fx_join(bb), s.kb, hig, s.kA, kd, m);
    }
};

// x 2^-d on the exponent's bits; 0 below the normal range
__device__ __forceinline__ double shift_down(double x, int d) {
    return biased_exp(x) <= d ? 0.0 : __hiloint2double(__double2hiint(x) - (d << 20), __double2loint(x));
}

// The pair loop in float64 for a CTA with an element out of range: inputs still float64 in shared memory.  One
// thread per line, the lines numbered consecutively over the threads: a float64 instruction costs its pipe 64
// clocks whatever its active lanes, and the half-filled last round of the cyclic distances would be a seventh
// (N = 8) to a third (N = 4) more of them.
template <int N>
__device__ __noinline__ void pairs_f64(double* smem, int n_el, const Ops& ops, const Phys& ph) {
    using C = AdjCfg<N>;
    constexpr int N2 = C::N2, SL = C::SL;
#pragma unroll 1
    for (int g = threadIdx.x; g < n_el * 3 * N2; g += C::THREADS) {
        const int e = g / (3 * N2), r = g - e * 3 * N2;
        const int l = r / N2, li = r - l * N2;
        const int c1 = li % N, c2 = li / N;
        double* se = smem + (size_t)e * C::SM;
        const double *X = se + C::XP, *n = se + C::XN + 3 * l * SL, *lt = se + C::LT;
        double* B = se + C::B + 6 * l * SL;
        auto prim = [&](int k) { return PrimH{2.0 * X[k], X[SL + k], X[2 * SL + k], X[3 * SL + k], X[4 * SL + k], X[5 * SL + k]}; };
        auto sums = [&](int k) { return PRaw{B[k], B[SL + k], B[2 * SL + k], B[3 * SL + k], B[4 * SL + k], B[5 * SL + k]}; };
        auto store = [&](int k, const PRaw& p) {
            B[k] = p.rho;
            B[SL + k] = p.u0;
            B[2 * SL + k] = p.u1;
            B[3 * SL + k] = p.u2;
            B[4 * SL + k] = p.beta;
            B[5 * SL + k] = p.c;
        };
        for (int i = 0; i < N; ++i) store(line_slot<N>(l, i, c1, c2), PRaw{0, 0, 0, 0, 0, 0});
#pragma unroll 1
        for (int i = 0; i < N - 1; ++i) {
            const int ii = line_slot<N>(l, i, c1, c2);
            const PrimH a = prim(ii);
            PRaw acc = sums(ii);
#pragma unroll 1
            for (int j = i + 1; j < N; ++j) {
                const int jj = line_slot<N>(l, j, c1, c2);
                PRaw o = sums(jj);
                double mu[5];
#pragma unroll
                for (int v = 0; v < 5; ++v)
                    mu[v] = ops.S[i][j] * (lt[v * SL + jj] * ops.winv[j] - lt[v * SL + ii] * ops.winv[i]);
                ec_pair_vjp(a, prim(jj), n[ii] + n[jj], n[SL + ii] + n[SL + jj], n[2 * SL + ii] + n[2 * SL + jj], mu, ph, acc, o);
                store(jj, o);
            }
            store(ii, acc);
        }
    }
}

template <int N>
__global__ void __launch_bounds__(AdjCfg<N>::THREADS, AdjCfg<N>::MINB)
adj_pairs_fix(const double* __restrict__ q, const double* __restrict__ lam, const double* __restrict__ geom,
              const double* __restrict__ jinv, double* __restrict__ pbar, int64_t K, const __grid_constant__ Ops ops,
              const __grid_constant__ Phys ph, const int32_t* __restrict__ kn) {
    using C = AdjCfg<N>;
    constexpr int N2 = C::N2, N3 = C::N3, EPB = C::EPB, SL = C::SL, NE = 11;
    extern __shared__ double smem[];
    __shared__ int sE[EPB][NE];
    __shared__ FixScale sScale[EPB];
    __shared__ AdjScale sAdj[EPB];
    __shared__ Fx sS[(N / 2) * N], sW[N];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int el_loc = t / N3, node = t - el_loc * N3;
    const int64_t el = (int64_t)blockIdx.x * EPB + el_loc;
    const bool active = el_loc < EPB && el < K;
    const int n_el = (int)(K - (int64_t)blockIdx.x * EPB < EPB ? K - (int64_t)blockIdx.x * EPB : EPB);
    double* sm = smem + (size_t)el_loc * C::SM;
    Fx* X = reinterpret_cast<Fx*>(sm);
    const int own = slot<N>(node % N, (node / N) % N, node / N2);
    for (int i = t; i < EPB * NE; i += C::THREADS)
        sE[i / NE][i % NE] = i % NE == 5 && i / NE < n_el ? kn[(int64_t)blockIdx.x * EPB + i / NE] : 0;
    for (int i = t; i < (N / 2) * N; i += C::THREADS) sS[i] = ops.SF[i / N][i % N];
    for (int i = t; i < N; i += C::THREADS) sW[i] = ops.WB[i];
    __syncthreads();
    if (active) {
        double qv[5], pi[6], RT;
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = q[(el * 5 + v) * N3 + node];
        const double Jinv = jinv[el * N3 + node];
        int E[NE];
        E[5] = 0;
#pragma unroll
        for (int c = 0; c < 9; ++c) sm[C::XN + c * SL + own] = geom[(el * 10 + 1 + c) * N3 + node];
        double lt[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            lt[v] = lam[(el * 5 + v) * N3 + node] * Jinv;
            sm[C::LT + v * SL + own] = lt[v];
        }
        // of lambda/(J w), with the node's largest 1/w of the three directions: lambda carries the weights, so a
        // bound by the end nodes' 1/w alone would leave the top bits empty
        const int we = max(ops.WE[node % N], max(ops.WE[(node / N) % N], ops.WE[node / N2]));
        int el_[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            const int b = biased_exp(lt[v]);
            el_[v] = b == 0 ? 0 : b + we;
        }
        E[6] = el_[0];
        E[7] = max(el_[1], max(el_[2], el_[3]));
        E[8] = el_[4];
        pair_inputs<kFluxESC>(qv, ph, pi, RT);
#pragma unroll
        for (int i = 0; i < 6; ++i) sm[C::XP + i * SL + own] = pi[i];
        pair_exponents<6>(pi, E);
        const int hp = double_hi(2.0 * pi[0] * RT);
        E[9] = hp;
        E[10] = 0x7ff00000 - hp;
        block_max<EPB == 1 || N3 % 32 == 0>(sE[el_loc], el_loc, E, lane);
    }
    __syncthreads();
    bool ok = true;
    for (int e = 0; e < n_el; ++e) {
        const int* E = sE[e];
        ok = ok && fix_range_ok(E[0], 4096 - E[1], E[2], E[3], 4096 - E[4], E[5]) && E[6] < 1151 && E[7] < 1151 && E[8] < 1151;
    }
    if (ok) {
        if (active) {
            const int* E = sE[el_loc];
            const FixScale s = fix_scale(E[0], 4096 - E[1], E[2], E[3], 4096 - E[4], E[5], 1000, 1000, ops.kg);
            const AdjScale ta = adj_scale(s, E[6], E[7], E[8], 0x7ff00000 - E[10], E[9]);
            if (node == 0) {
                sScale[el_loc] = s;
                sAdj[el_loc] = ta;
            }
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                const int i = C::XN + c * SL + own;
                X[i] = fx_split(fx_from_double(sm[i], s.kn));
            }
            scale_inputs<kFluxESC>(sm + C::XP + own, X + C::XP + own, SL, s);
        }
        __syncthreads();
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
            const Fx* Xe = reinterpret_cast<const Fx*>(se);
            const Fx *XP = Xe + C::XP, *XN = Xe + C::XN + 3 * l * SL;
            const FixScale& s = sScale[e];
            const AdjScale& ta = sAdj[e];
            const int ic = i < N ? i : 0, ii = line_slot<N>(l, ic, c1, c2);
            const PrimFx a = load_inputs<kFluxESC>(XP + ii, SL);
            const Fx na0 = XN[ii], na1 = XN[SL + ii], na2 = XN[2 * SL + ii], w = sW[ic];
            // lambda/(J w) in fixed point, shifted up by what the line's largest leaves free of the element's bound
            double lt[5];
            int up = 60;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                lt[v] = se[C::LT + v * SL + ii];
                const int b = biased_exp(lt[v]);
                if (b) up = min(up, sE[e][v == 0 ? 6 : (v == 4 ? 8 : 7)] - b - ops.WE[ic]);
            }
            const int mine = up;
#pragma unroll
            for (int k = 1; k < N; ++k) up = min(up, __shfl_sync(0xffffffffu, mine, (lw * N + (ic + k < N ? ic + k : ic + k - N)) & 31));
            long long lo[5];
#pragma unroll
            for (int v = 0; v < 5; ++v)
                lo[v] = fx_mul(fx_split(fx_from_double(lt[v], (v == 0 ? ta.l0 : (v == 4 ? ta.l4 : ta.l1)) - ops.kW - up)), w);
            PairBarFx acc = {0.0, 0.0, 0.0, 0.0, {0.0, 0.0, 0.0}, 0.0};
#pragma unroll 1
            for (int k = 1; k <= N / 2; ++k) {
                const int j = ic + k < N ? ic + k : ic + k - N;
                const int to = (lw * N + j) & 31;
                long long mu[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) mu[v] = __shfl_sync(0xffffffffu, lo[v], to) - lo[v];
                PairBarFx o = {0.0, 0.0, 0.0, 0.0, {0.0, 0.0, 0.0}, 0.0};
                if (go && (2 * k < N || i < k)) {
                    const int jj = line_slot<N>(l, j, c1, c2);
                    const PrimFx b = load_inputs<kFluxESC>(XP + jj, SL);
                    const Fx S = sS[(k - 1) * N + i];
                    const Fx n0 = fx_split(fx_mul<2>(S, fx_add(na0, XN[jj]))), n1 = fx_split(fx_mul<2>(S, fx_add(na1, XN[SL + jj]))),
                             n2 = fx_split(fx_mul<2>(S, fx_add(na2, XN[2 * SL + jj])));
                    const AdjMeansF64 lm = {a.r, b.r, a.b, b.b, s, ta.kd, 0.5 * ph.inv_gm1};
                    ec_pair_vjp_fx(a, b, n0, n1, n2, mu, ops.CG, s, ta, lm, o);
                    acc.xa += o.xa;
                    acc.ba += o.ba;
                    acc.c += o.c;
#pragma unroll
                    for (int d = 0; d < 3; ++d) acc.u[d] += o.u[d];
                }
                const int from = (lw * N + (i >= k ? i - k : i - k + N)) & 31;
                acc.xa += __shfl_sync(0xffffffffu, o.xb, from);
                acc.ba += __shfl_sync(0xffffffffu, o.bb, from);
                acc.c += __shfl_sync(0xffffffffu, o.c, from);
#pragma unroll
                for (int d = 0; d < 3; ++d) acc.u[d] += __shfl_sync(0xffffffffu, o.u[d], from);
            }
            if (go) {
                double* B = se + C::B + 6 * l * SL + ii;
                B[0] = shift_down(acc.xa, up);
#pragma unroll
                for (int d = 0; d < 3; ++d) B[(1 + d) * SL] = shift_down(acc.u[d], up);
                B[4 * SL] = shift_down(acc.ba, up);
                B[5 * SL] = shift_down(acc.c, up);
            }
        }
    } else {
        pairs_f64<N>(smem, n_el, ops, ph);
    }
    __syncthreads();
    if (active) {
        // sums of the directions; r[0] = rho rho-bar + beta beta-bar
        double r[6], qv[5], RT;
        Prim p;
#pragma unroll
        for (int v = 0; v < 5; ++v) qv[v] = q[(el * 5 + v) * N3 + node];
        to_prim_fx(qv, ph, p, RT);
        const double* B = sm + C::B + own;
#pragma unroll
        for (int c = 0; c < 6; ++c) r[c] = B[c * SL] + B[(6 + c) * SL] + B[(12 + c) * SL];
        if (!ok) r[0] = fma(p.beta, r[4], qv[0] * r[0]);
        // to the conserved variables: beta = rho/(2p), p-bar = -2 beta^2/rho beta-bar, |u|^2-bar = -c/4
        const double ri = rcp_cubic(qv[0]);
        const double pb = -2.0 * p.beta * p.beta * ri * r[4] * ph.gm1;
        const double w0 = fma(-r[5], p.hu0, 0.5 * r[1]), w1 = fma(-r[5], p.hu1, 0.5 * r[2]), w2 = fma(-r[5], p.hu2, 0.5 * r[3]);
        double* o = pbar + el * 5 * N3 + node;
        o[0] = fma(ri, r[0] - 2.0 * fma(w2, p.hu2, fma(w1, p.hu1, w0 * p.hu0)), 2.0 * pb * p.qq);
        o[N3] = fma(w0, ri, -2.0 * pb * p.hu0);
        o[2 * N3] = fma(w1, ri, -2.0 * pb * p.hu1);
        o[3 * N3] = fma(w2, ri, -2.0 * pb * p.hu2);
        o[4 * N3] = pb;
    }
}

template <int N>
cudaError_t prepare_n_adj() {
    return cudaFuncSetAttribute(adj_pairs_fix<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(AdjCfg<N>::EPB * AdjCfg<N>::SM * sizeof(double)));
}
template <int N>
cudaError_t launch_n_adj(const esdc_ctx* c, const double* q, const double* lam, cudaStream_t s) {
    using C = AdjCfg<N>;
    adj_pairs_fix<N><<<(unsigned)((c->K + C::EPB - 1) / C::EPB), C::THREADS, C::EPB * C::SM * sizeof(double), s>>>(
        q, lam, c->d_geom, c->d_jinv, c->d_adj_pb, c->K, c->ops, c->phys, c->d_kn);
    return cudaGetLastError();
}

}  // namespace

cudaError_t prepare_adj_pairs(const esdc_ctx* c) {
    switch (c->N) {
        case 2: return prepare_n_adj<2>();
        case 3: return prepare_n_adj<3>();
        case 4: return prepare_n_adj<4>();
        case 5: return prepare_n_adj<5>();
        case 6: return prepare_n_adj<6>();
        case 7: return prepare_n_adj<7>();
        case 8: return prepare_n_adj<8>();
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_adj_pairs(const esdc_ctx* c, const double* q, const double* lam, cudaStream_t s) {
    switch (c->N) {
        case 2: return launch_n_adj<2>(c, q, lam, s);
        case 3: return launch_n_adj<3>(c, q, lam, s);
        case 4: return launch_n_adj<4>(c, q, lam, s);
        case 5: return launch_n_adj<5>(c, q, lam, s);
        case 6: return launch_n_adj<6>(c, q, lam, s);
        case 7: return launch_n_adj<7>(c, q, lam, s);
        case 8: return launch_n_adj<8>(c, q, lam, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace esdc
