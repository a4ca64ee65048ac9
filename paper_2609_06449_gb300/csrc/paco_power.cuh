// paco_power.cuh -- the two stages of the weighted power of the spectrum
// (complex64): Phase I with the redistribution in its stores, and Phase III
// with sum w |y|^2 over its results, each over the plan's own factors.
//
// A tile of W columns of an L-row view per CTA, L = A * B with both factors in
// registers (j = j_hi B + j_lo, k = k_lo + A k_hi): A-point DFTs over j_hi,
// w_L^{-k_lo j_lo}, one exchange through shared memory, B-point DFTs over j_lo.
// Strides are launch arguments, all else is fixed at compile time; row maps are
// bit permutations (pi in any base 2^t is one), so the row of j is the sum of a
// per-thread term for j_lo and one of at most 32 launch constants for j_hi.
//
// Measured on GB300, 256 x 2^20 with the sum: 3.34 -> 1.86 ms against the generic
// stage kernels, which spend 130-140 warp instructions a point on run-time
// strides and twiddle products.
#pragma once

#include "../../include/paco.h"
#include "paco_fold.cuh"

namespace paco {

struct PowerArgs {
    const cx<float> *in;
    cx<float> *out;
    long long bstride;      // elements between two transforms (input and output)
    unsigned rowA[32];      // element offset of input row (j_hi B) under the row map
    unsigned rowK[32];      // Phase III: element offset of output row A k_hi
    unsigned ld_in, ld_out; // elements between two rows
    int rev_bits, rev_t;    // row map of j_lo: pi over rev_bits bits (0: natural rows)
    int crev_bits, crev_t;  // Phase I: row pi(c) of column c
    int lg_all;             // log2 of the tiles of one transform (blockIdx.x = transform, tile)
    const cx<float> *twL;   // w_L^{-r}, r < L, as the stage kernels' product of two factors (plan_tables)
    const cx<float> *lo;    // w_N^{-r}, r < 2^lo_bits
    const cx<float> *hi;    // w_N^{-(r << lo_bits)}
    int lo_bits;
    unsigned n_mask;        // N - 1
    int conj;               // 1: the conjugate transform
    int reverse;            // 1: tiles from the last to the first (what the pass before wrote last is in L2)
    const float *w;         // Phase III: *loss += sum over n of w[n] |out[n]|^2, and
    double *loss;
    int store_weighted;     //   (1) w[n] * out[n] is stored in place of out[n]
};

// ---- the stage kernels' arithmetic, operation by operation ------------------
// The weighted power is summed in 64 bits over a whole batch: roundings that
// follow the data average out, but those of twiddle products and constants do
// not, and another sequence of equally accurate operations moves the sum by
// 1e-9 to 1e-7 of its value.  These kernels therefore state each
// fused multiply-add explicitly, in the order paco_stage.cuh's kernels compile
// to (found by comparing their results bit by bit), so that the sum does not
// depend on which kernel ran a stage.
namespace st {

// a * b with one product of each part fused: YO picks which one of the imaginary part
template <int YO>
__device__ __forceinline__ cx<float> mul(cx<float> a, cx<float> b)
{
    return make_cx<float>(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)),
                          YO ? __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)) : __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
// a +- h p
__device__ __forceinline__ cx<float> axpy(cx<float> a, float h, cx<float> p)
{
    return make_cx<float>(__fmaf_rn(h, p.x, a.x), __fmaf_rn(h, p.y, a.y));
}
constexpr float H = PACO_RH, C8 = PACO_C8, S8 = PACO_S8;
__device__ __forceinline__ cx<float> w8_1(cx<float> a) { return make_cx<float>(a.x + a.y, a.y - a.x); }     // times H
__device__ __forceinline__ cx<float> w8_3(cx<float> a) { return make_cx<float>(a.y - a.x, -(a.x + a.y)); }  // times H

__device__ __forceinline__ void dft8(cx<float> *v)
{
    using C = cx<float>;
    C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4(e);
    dft4(o);
    const C p1 = w8_1(o[1]), p2 = mul_mi(o[2]), p3 = w8_3(o[3]);
    v[0] = e[0] + o[0]; v[4] = e[0] - o[0];
    v[1] = axpy(e[1], H, p1); v[5] = axpy(e[1], -H, p1);
    v[2] = e[2] + p2; v[6] = e[2] - p2;
    v[3] = axpy(e[3], H, p3); v[7] = axpy(e[3], -H, p3);
}

__device__ __forceinline__ void dft16(cx<float> *v)
{
    using C = cx<float>;
#pragma unroll
    for (int r = 0; r < 4; ++r) dft4_s(v[r], v[r + 4], v[r + 8], v[r + 12]);
    const C v5 = mul<1>(v[5], make_cx<float>(C8, -S8)), v13 = mul<1>(v[13], make_cx<float>(S8, -C8));
    const C v7 = mul<1>(v[7], make_cx<float>(S8, -C8)), v15 = mul<0>(v[15], make_cx<float>(-C8, S8));
    const C p9 = w8_1(v[9]), p6 = w8_1(v[6]), p14 = w8_3(v[14]), p11 = w8_3(v[11]), v10 = mul_mi(v[10]);
    C y[16];
    auto row = [&](int s, C t0, C t1, C t2, C d) {        // d = v1 - v3
        const C t3 = mul_mi(d);
        y[s] = t0 + t2; y[s + 8] = t0 - t2; y[s + 4] = t1 + t3; y[s + 12] = t1 - t3;
    };
    row(0, v[0] + v[2], v[0] - v[2], v[1] + v[3], v[1] - v[3]);
    row(1, axpy(v[4], H, p6), axpy(v[4], -H, p6), v5 + v7, v5 - v7);
    const C m11 = make_cx<float>(__fmul_rn(H, p11.x), __fmul_rn(H, p11.y));
    row(2, v[8] + v10, v[8] - v10, axpy(m11, H, p9), axpy(make_cx<float>(-m11.x, -m11.y), H, p9));
    row(3, axpy(v[12], H, p14), axpy(v[12], -H, p14), v13 + v15, v13 - v15);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = y[k];
}

// 16 x 2 with w_32 as a general product
__device__ __forceinline__ void dft32(cx<float> *v)
{
    constexpr float c[9] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                            0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                            0.19509032201612826785f, 0.f};
    cx<float> e[16], o[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        e[r] = v[2 * r];
        o[r] = v[2 * r + 1];
    }
    dft16(e);
    dft16(o);
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        // w_32^{-s} = cos - i sin, sin(s) = cos(|8 - s|)
        const cx<float> w = make_cx<float>(s <= 8 ? c[s] : -c[16 - s], -c[s <= 8 ? 8 - s : s - 8]);
        const cx<float> t = s > 0 ? mul<1>(o[s], w) : o[s];
        v[s] = e[s] + t;
        v[s + 16] = e[s] - t;
    }
}

} // namespace st

template <int RADIX>
__device__ __forceinline__ void st_dft(cx<float> *v)
{
    if constexpr (RADIX == 32) st::dft32(v);
    else if constexpr (RADIX == 16) st::dft16(v);
    else if constexpr (RADIX == 8) st::dft8(v);
    else dft<RADIX>(v);
}

// w_N^{-r} from the two-level table.
__device__ __forceinline__ cx<float> st_tw_n(const PowerArgs &a, unsigned r)
{
    const float2 l = __ldg(reinterpret_cast<const float2 *>(a.lo + (r & ((1u << a.lo_bits) - 1u))));
    const float2 h = __ldg(reinterpret_cast<const float2 *>(a.hi + (r >> a.lo_bits)));
    return st::mul<0>(make_cx<float>(l.x, l.y), make_cx<float>(h.x, h.y));
}

template <int LGA_, int LGB_, int LGW_, bool FIRST_>
struct PowerCfg {
    static constexpr int LGA = LGA_, LGB = LGB_, LGW = LGW_;
    static constexpr bool FIRST = FIRST_;
    static constexpr int A = 1 << LGA, B = 1 << LGB, W = 1 << LGW, L = A * B;
    static constexpr int EPT = (LGA == 5 || LGB == 5) ? 32 : 16;   // points a thread holds
    static constexpr int NT = L * W / EPT;
    static constexpr int U1 = EPT / A, U2 = EPT / B;               // sequences a thread, F1 and F2
    // Exchange layouts (in points).  FIRST: [col][j_lo][k_lo], F2 reads runs of
    // k_lo; else [k_lo][j_lo][col], F2 reads runs of columns.  The pads make
    // every half-warp of 8-byte accesses on either side hit 16 different banks.
    static constexpr int SJ = FIRST ? A + 1 : W;
    static constexpr int SC0 = B * SJ;
    static constexpr int SC = FIRST ? SC0 + (((W < 16 ? 16 / W : 1) - SC0 % 16 + 16) % 16) : 1;
    static constexpr int SK = FIRST ? 1 : B * W + (W < 16 ? (W - (B * W) % 16 + 16) % 16 : 0);
    static constexpr int EX = FIRST ? W * SC : A * SK;
    static constexpr int NTW = FIRST ? B * W : 0;                  // per-tile twiddles
    static constexpr int SMEM = (EX + NTW) * 8;
    static constexpr int REGS_CTAS = (EPT == 32 ? 512 : 1024) / NT;
    static constexpr int SMEM_CTAS = (227 * 1024) / (SMEM + 1024);
    static constexpr int MINB = REGS_CTAS < 1 ? 1 : (REGS_CTAS < SMEM_CTAS ? REGS_CTAS : SMEM_CTAS);
};

template <class CFG>
__global__ void __launch_bounds__(CFG::NT, CFG::MINB) paco_power_kernel(const __grid_constant__ PowerArgs a)
{
    using C = cx<float>;
    constexpr int A = CFG::A, B = CFG::B, W = CFG::W, EPT = CFG::EPT, NT = CFG::NT;
    constexpr int U1 = CFG::U1, U2 = CFG::U2;
    constexpr bool FIRST = CFG::FIRST;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    C *tab = sm + CFG::EX;
    const int tid = threadIdx.x;
    grid_launch_dependents();
    const unsigned bid = a.reverse ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
    const long long boff = (long long)(bid >> a.lg_all) * a.bstride;
    const unsigned c0 = (bid & ((1u << a.lg_all) - 1u)) << CFG::LGW;
    const long long base = boff + c0;
    const float sg = a.conj ? -1.f : 1.f;

    grid_wait();
    // ---- F1
    C v[EPT];
#pragma unroll
    for (int u = 0; u < U1; ++u) {
        const int s = tid + NT * u, col = s & (W - 1), jlo = s >> CFG::LGW;
        const unsigned jrow = a.rev_bits ? digit_reverse((unsigned)jlo, a.rev_bits, a.rev_t) : (unsigned)jlo;
        const float2 *p = reinterpret_cast<const float2 *>(a.in + base + col + (long long)jrow * a.ld_in);
#pragma unroll
        for (int r = 0; r < A; ++r) {
            const float2 t = ld_data(p + a.rowA[r]);
            v[u * A + r] = make_cx<float>(t.x, t.y * sg);
        }
    }
    // the tile's twiddles w_N^{-A k_hi c}, [k_hi][col], under the loads' latency
    if constexpr (FIRST) {
#pragma unroll
        for (int e = tid; e < B * W; e += NT) {
            const unsigned c = c0 + (e & (W - 1));
            tab[e] = st_tw_n(a, ((unsigned)(e >> CFG::LGW) * (unsigned)A * c) & a.n_mask);
        }
    }
    const float2 *tw = reinterpret_cast<const float2 *>(a.twL);
#pragma unroll
    for (int u = 0; u < U1; ++u) {
        const int s = tid + NT * u, col = s & (W - 1), jlo = s >> CFG::LGW;
        st_dft<A>(v + u * A);
        C *ex = sm + (FIRST ? col * CFG::SC + jlo * CFG::SJ : jlo * W + col);
        ex[0] = v[u * A];
#pragma unroll
        for (int k = 1; k < A; ++k) {
            const float2 t = __ldg(tw + k * jlo);
            ex[FIRST ? k : k * CFG::SK] = st::mul<0>(v[u * A + k], make_cx<float>(t.x, t.y));
        }
    }
    // w_N^{-k_lo c} (read before the barrier: its two table reads overlap the others' F1)
    [[maybe_unused]] C e1[U2];
    if constexpr (FIRST) {
#pragma unroll
        for (int u = 0; u < U2; ++u) {
            const int s = tid + NT * u;
            e1[u] = st_tw_n(a, ((unsigned)(s & (A - 1)) * (c0 + (unsigned)(s >> CFG::LGA))) & a.n_mask);
        }
    }
    __syncthreads();

    // ---- F2.  A thread's float sums run over 16 results each, grouped as in
    // the stage kernels (32 results of one sequence: those of even and of odd k_hi).
    constexpr int NP = EPT / 16;
    [[maybe_unused]] float power[NP] = {};
#pragma unroll
    for (int u = 0; u < U2; ++u) {
        const int s = tid + NT * u;
        int col, klo;
        if constexpr (FIRST) { klo = s & (A - 1); col = s >> CFG::LGA; }
        else { col = s & (W - 1); klo = s >> CFG::LGW; }
        const C *ex = sm + (FIRST ? col * CFG::SC + klo : klo * CFG::SK + col);
#pragma unroll
        for (int r = 0; r < B; ++r) v[u * B + r] = ex[r * CFG::SJ];
        st_dft<B>(v + u * B);
        if constexpr (FIRST) {
#pragma unroll
            for (int k = 0; k < B; ++k)
                v[u * B + k] = st::mul<0>(v[u * B + k], st::mul<1>(e1[u], tab[(k << CFG::LGW) + col]));
            const unsigned c = c0 + col;
            const unsigned row = a.crev_bits ? digit_reverse(c, a.crev_bits, a.crev_t) : c;
            float2 *q = reinterpret_cast<float2 *>(a.out + boff + (long long)row * a.ld_out + klo);
#pragma unroll
            for (int k = 0; k < B; ++k) q[A * k] = make_float2(v[u * B + k].x, v[u * B + k].y * sg);
        } else {
            const long long o = base + col + (long long)klo * a.ld_out;
            // k_hi in the order 0, 16, 2, 18, ..., 14, 30, then 1, 17, ... for B = 32;
            // the weights of 16 results at a time (32 would not fit the registers)
            constexpr int H = B < 16 ? B : 16;
#pragma unroll
            for (int g = 0; g < B / H; ++g) {
                float wv[H];
#pragma unroll
                for (int i = 0; i < H; ++i)
                    wv[i] = ld_data(a.w + o + a.rowK[B == 32 ? g + 2 * (i >> 1) + 16 * (i & 1) : i]);
                float &pw = power[B == 32 ? g : NP == 1 ? 0 : u];
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    C &y = v[u * B + (B == 32 ? g + 2 * (i >> 1) + 16 * (i & 1) : i)];
                    pw = __fmaf_rn(wv[i], __fmaf_rn(y.x, y.x, __fmul_rn(y.y, y.y)), pw);
                    if (a.store_weighted) y = make_cx<float>(y.x * wv[i], y.y * wv[i]);
                }
            }
            float2 *q = reinterpret_cast<float2 *>(a.out + o);
#pragma unroll
            for (int k = 0; k < B; ++k) q[a.rowK[k]] = make_float2(v[u * B + k].x, v[u * B + k].y * sg);
        }
    }
    if constexpr (!FIRST) {
        // warp sums, then one FP64 atomic a CTA
        double *wsum = reinterpret_cast<double *>(sm);
        __syncthreads();                                  // every read of the exchange is done
#pragma unroll
        for (int i = 0; i < NP; ++i) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) power[i] += __shfl_xor_sync(0xffffffffu, power[i], o);
            if ((tid & 31) == 0) wsum[i * (NT / 32) + (tid >> 5)] = (double)power[i];
        }
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int i = 0; i < NP * (NT / 32); ++i) t += wsum[i];
            atomicAdd(a.loss, t);
        }
    }
}

// What the host needs to launch one of the kernels above.
struct PowerKernel {
    const void *fn = nullptr;
    int lgA = 0, lgB = 0, lgW = 0, threads = 0, smem = 0;
};

// The kernel of a stage of length 2^lgL over 2^lgC columns; fn == nullptr
// where none is built.
PowerKernel power_kernel(bool first, int lgL, int lgC);

} // namespace paco
