// paco_whole.cuh -- whole complex64 transforms of up to 2^14 points in one CTA.
//
// A CTA holds NT EPT points, as many transforms as fit; they cross memory once
// in each direction (16 B a point) where two passes take 32.  Two or three
// register steps of radix up to 32 find the frequencies digit by digit, most
// significant input digit first: before a step K of them are known, a sequence
// is (kappa in [K], j_lo), and its DFT over the next digit takes the folded
// twiddles of paco_fold.cuh, so that Phase I, the redistribution of Sect. 4.2
// and Phase III are one chain of exchanges in shared memory and all pairs of
// the paper's exchange are self pairs.  Loads are runs of j_lo, stores runs of
// kappa, of at least 64 bytes from 2^6 points on.
//
// Exchange layout: point (kappa', j_lo) of transform g at
// g GS + kappa' + (K' + 1) j_lo, K' the frequencies known after the step: a
// half-warp writes 16 j_lo (odd stride) or 16 kappa and reads 16 kappa' or
// 8 + 8 -- 16 different banks (4-point rows aside).
#pragma once

#include "paco_fold.cuh"

namespace paco {

// The radix of step i of 2^lg points (0: no such step), 4 <= lg <= 14.
__host__ __device__ constexpr int whole_radix(int lg, int i)
{
    constexpr int table[11][3] = {{4, 4, 0}, {8, 4, 0}, {8, 8, 0}, {8, 16, 0}, {16, 16, 0}, {8, 8, 8},
                                  {16, 8, 8}, {16, 16, 8}, {16, 16, 16}, {32, 16, 16}, {32, 32, 16}};
    return i < 3 ? table[lg - 4][i] : 0;
}

template <int LG>
struct WholeSteps {
    static constexpr int r(int i) { return whole_radix(LG, i); }
    static constexpr int k(int i) { return i == 0 ? 1 : k(i - 1) * r(i - 1); }      // frequencies known before step i
    static constexpr int N = 1 << LG;
    static constexpr int tau(int i) { return i <= 1 ? 0 : tau(i - 1) + k(i - 1) * r(i - 1) / 2; }   // step i's factors
    static constexpr int TAU = r(2) ? tau(2) + k(2) * r(2) / 2 : k(1) * r(1) / 2;
    static constexpr int rows(int i) { return N / k(i + 1); }                       // j_lo left after step i
    static constexpr int gs(int i)                                                  // exchange after step i
    {
        const int b = rows(i) * (k(i + 1) + 1);
        return k(i + 1) < 16 ? (b + 7) / 16 * 16 + 8 : b;
    }
};

// DIRECT_FROM: the length from which the butterflies are DIRECT (whole_step).
template <int LG_, int EPT, int NT, int DIRECT_FROM = 8192>
struct WholeCfg {
    using S = WholeSteps<LG_>;
    static constexpr int LG = LG_, N = 1 << LG, TE = EPT * NT, G = TE / N;
    static constexpr int EX0 = G * S::gs(0), EX1 = S::r(2) ? G * S::gs(1) : 0;
    static constexpr int SMEM = (EX0 > EX1 ? EX0 : EX1) * 8;
    static constexpr bool CARRIES = N > 128 && N < DIRECT_FROM;    // CARRY butterflies
    static_assert(G >= 1 && S::r(0) <= EPT, "tile");
};

// Step I of the tile's transforms.  off(g): element offset of transform g, or
// negative where the tile has none; SCALED: f multiplies the input (as a branch in
// the one kernel it cost every other call: 2^12 points 0.641 -> 0.650 ms per 2^28).
// True: nothing was stored, the tile is to be done with AGAIN (may_overflow).
template <class CFG, int EPT, int NT, int I, bool SCALED, bool AGAIN = false, class Off>
__device__ __forceinline__ bool whole_step(const float2 *in, float2 *out, bool conj, float f, const float2 *tau,
                                           const Off &off, cx<float> *sm)
{
    using S = typename CFG::S;
    using C = cx<float>;
    constexpr int R = S::r(I), K = S::k(I), N = CFG::N, SQ = N / R, U = EPT / R, J = SQ / K;
    constexpr bool LAST = S::r(I + 1) == 0;
    // Up to 2^7 points the copy rate leaves room for the closer form.  Above, the
    // question (may_overflow) costs less: 2^12 points 0.641 ms per 2^28 without it, 0.642
    // with it, DIRECT 0.655; but not with 32 points a thread: 2^13 0.698, 0.757, 0.737, 2^14
    // 0.930, 0.953, 0.945 (the uneven batch keeps the question there, DIRECT spills).
    constexpr int KIND = AGAIN ? SAFE : !CFG::CARRIES ? DIRECT : CARRY;
    const int tid = threadIdx.x;
    C v[EPT];
    [[maybe_unused]] bool big = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int s = tid + NT * u, g = s / SQ, idx = s % SQ;
        if constexpr (I == 0) {
            const long long o = off(g);
            const float2 *p = in + o + idx;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 t = o >= 0 ? __ldcg(p + r * SQ) : make_float2(0.f, 0.f);
                v[u * R + r] = make_cx<float>(t.x, t.y);
            }
        } else {
            const C *p = sm + g * S::gs(I - 1) + idx % K + (K + 1) * (idx / K);
#pragma unroll
            for (int r = 0; r < R; ++r) v[u * R + r] = p[(K + 1) * J * r];
        }
    }
    if constexpr (I > 0 && !LAST) __syncthreads();        // read before the next exchange overwrites it
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int s = tid + NT * u, g = s / SQ, idx = s % SQ, kap = idx % K, jlo = idx / K;
        if constexpr (I == 0) {
            // the conjugate transform as the forward one of (im, re), swapped back at the end
            if (conj) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[u * R + r] = make_cx<float>(v[u * R + r].y, v[u * R + r].x);
            }
            if constexpr (SCALED) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[u * R + r] = make_cx<float>(v[u * R + r].x * f, v[u * R + r].y * f);
            }
            if constexpr (KIND == CARRY) big |= may_overflow<R>(v + u * R, CFG::LG);
            plain_dft<R>(v + u * R);
        } else {
            fold_dft<KIND, float, R>(v + u * R, [&](int q) {
                const float2 t = __ldg(tau + S::tau(I) + q * K + kap);
                return make_cx<float>(t.x, t.y);
            });
        }
        if constexpr (!LAST) {
            C *p = sm + g * S::gs(I) + kap + (K * R + 1) * jlo;
#pragma unroll
            for (int k = 0; k < R; ++k) p[K * k] = v[u * R + k];
        } else {
            const long long o = off(g);
            if (o >= 0) {
                float2 *q = out + o + kap;
                if (conj) {
#pragma unroll
                    for (int k = 0; k < R; ++k) q[K * k] = make_float2(v[u * R + k].y, v[u * R + k].x);
                } else {
#pragma unroll
                    for (int k = 0; k < R; ++k) q[K * k] = make_float2(v[u * R + k].x, v[u * R + k].y);
                }
            }
        }
    }
    if constexpr (!LAST) {
        if constexpr (I == 0 && KIND == CARRY) {
            if (__syncthreads_or(big)) return true;
        } else {
            __syncthreads();
        }
        whole_step<CFG, EPT, NT, I + 1, SCALED, AGAIN>(in, out, conj, f, tau, off, sm);
    }
    return false;
}

// The tile with AGAIN, out of line: it takes no register of the common path.
template <class CFG, int EPT, int NT, bool SCALED, class Off>
__device__ __noinline__ void whole_again(const float2 *in, float2 *out, bool conj, float f, const float2 *tau, Off off,
                                         cx<float> *sm)
{
    whole_step<CFG, EPT, NT, 0, SCALED, true>(in, out, conj, f, tau, off, sm);
}

// The tile's transforms, again where they may overflow.
template <class CFG, int EPT, int NT, bool SCALED, class Off>
__device__ __forceinline__ void whole_tile(const float2 *in, float2 *out, bool conj, float f, const float2 *tau,
                                           const Off &off, cx<float> *sm)
{
    if (whole_step<CFG, EPT, NT, 0, SCALED>(in, out, conj, f, tau, off, sm)) {
        if constexpr (CFG::CARRIES) whole_again<CFG, EPT, NT, SCALED>(in, out, conj, f, tau, off, sm);
    }
}

struct WholeArgs {
    const float2 *in;
    float2 *out;
    long long batch;
    const float2 *tau;      // the steps' factors (WholeSteps::TAU entries)
    int conj;
    float mult;             // SCALED: the input is scaled by mult * (*scale or 1)
    const double *scale;
};

template <int LG, int EPT, int NT, bool SCALED>
__global__ void __launch_bounds__(NT, (EPT == 16 ? 1024 : 512) / NT) paco_whole_kernel(const __grid_constant__ WholeArgs a)
{
    using CFG = WholeCfg<LG, EPT, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const long long t0 = (long long)blockIdx.x * CFG::G;
    const float f = SCALED ? (a.scale ? a.mult * (float)__ldg(a.scale) : a.mult) : 1.f;
    whole_tile<CFG, EPT, NT, SCALED>(
        a.in, a.out, a.conj != 0, f, a.tau, [&](int g) { return t0 + g < a.batch ? (t0 + g) << LG : -1ll; },
        reinterpret_cast<cx<float> *>(smem_raw));
}

// The kernel for transforms of 2^lgN points, 4 <= lgN <= 14.
struct WholeKernel {
    const void *fn = nullptr;
    int threads = 0, smem = 0, per_cta = 0;
};
WholeKernel whole_kernel(int lgN, bool scaled);

// The factors of 2^lgN points (device table, paco_route.cu).
paco_status_t whole_table(int lgN, void **dst);

} // namespace paco
