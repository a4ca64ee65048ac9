// paco_fold.cuh -- a local-FFT pass with the inter-pass twiddles inside its
// butterflies.
//
// A transform of N points taken digit by digit, most significant input digit
// first, needs at every radix-2 level one factor per butterfly,
// w_{2M}^{-kappa} with M the number of frequencies found so far and kappa in
// [M] this one's index.  Written as
//     p = E + t O   (four fused multiply-adds),   E - t O = 2 E - p   (two)
// a level costs three operations a point, twiddle included, against the 2.6 of
// a radix-16 or -32 DFT plus the four of a separate complex product; nothing
// is multiplied on its way out of a pass, so Phase I stores plain DFTs and the
// top-level twiddle w_N^{-k1 c} (Sect. 3.3) is taken by Phase III's
// butterflies.  In complex128, which the FP64 pipe bounds, the count is the
// time (2^27: 27.5 ms with separate products in the stage kernels, 22.5 ms here).
// In complex64 it is the issue rate: a pass of 1024 points over 2^28 went from
// 1.38 ms (139 instructions a point) to 0.79.
//
// 2 E - p takes E - t O along where p overflows.  Tiles of such butterflies
// therefore ask whether their values are that large (may_overflow), and are done
// again with butterflies whose parts overflow each on its own; or the difference
// is computed directly, four operations a point and level (Bfly, FoldCfg::BFLY1
// and BFLY2).
//
// A pass transforms L = A B rows (j = j_hi B + j_lo, k = k_lo + A k_hi) of a
// tile of W columns: A-point DFTs over j_hi in registers, one exchange through
// shared memory, B-point DFTs over j_lo.  FIRST: kappa = 0, column c of the
// view is stored as row pi(c) of the result (the one redistribution).  Else
// the pass runs in place on row blocks, its columns are the frequencies found
// so far (kappa = column, K of them), and rows are read through pi.
//
// Twiddles (TW).  0: kappa = 0 (the first pass; every pass of the 2-D and 3-D
// forms).  1: all of the pass's factors come, rounded once from FP64, out of one
// table of about K L / 2 entries, a level's factors being a run in kappa.  2,
// where that table would not stay in L2 (K L > 2^20): the table holds F1's
// factors and w_{K L}^{-kappa 2^i}, a tile's part of which goes to shared memory,
// and a factor of F2 is one more product of such a value with w_L's.
//
// The folded butterflies multiply at every level, so the rounding of their
// factors shows: with all factors as products of rounded values the relative
// error of 2^24 points is 2.2e-7, with the tables above 1.9e-7 (the stage
// kernels: 2.0e-7).  2 E - p carries p's rounding on; in FP64, whose error is
// held to the stage kernels' too, F1 therefore multiplies its rows first and
// takes the plain DFT (ROWS), and F2 is direct from three passes on.
#pragma once

#include "../../include/paco.h"
#include "paco_common.cuh"

namespace paco {

template <typename R>
struct FoldArgs {
    const cx<R> *in;
    cx<R> *out;
    long long bstride;      // elements between two transforms
    unsigned rowA[32];      // element offset of input row (j_hi B) under the row map
    unsigned rowK[32];      // element offset of output row A k_hi (not FIRST)
    unsigned ld_in, ld_out; // elements between two rows
    int rev_bits, rev_t;    // row map of j_lo: pi over rev_bits bits (0: natural rows)
    int crev_bits, crev_t;  // FIRST: row pi(c) of column c
    int lg_tiles;           // log2 of the column tiles of one row block
    int lg_all;             // log2 of the tiles of one transform
    unsigned blk_stride;    // elements between two row blocks
    const cx<R> *tau;       // the factors (fold_table)
    int lg_n, lg_k;         // log2 N, log2 K
    int conj;               // 1: the conjugate transform
    int reverse;            // 1: tiles from the last to the first
    R mult;                 // SCALED: the input is scaled by mult * (*scale or 1)
    const double *scale;
};

template <typename R> struct vec2;
template <> struct vec2<float> { using type = float2; };
template <> struct vec2<double> { using type = double2; };

__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }

// (e, o) -> (e + t o, e - t o).
// CARRY: the second as 2 e - (e + t o).
// DIRECT: on its own, two more operations; the first one's rounding is not carried on.
// SAFE: where a sum may overflow.  CARRY then takes the finite difference beside
// an overflowing sum with it, and a product with a zero part of t makes a NaN of
// an infinite o: here each part overflows on its own.
enum Bfly { CARRY, DIRECT, SAFE };
template <int KIND, typename R>
__device__ __forceinline__ void bfly(cx<R> &e, cx<R> &o, cx<R> t)
{
    if constexpr (KIND == SAFE) {
        cx<R> m;
        if (t.y == R(0)) m = make_cx<R>(t.x * o.x, t.x * o.y);
        else if (t.x == R(0)) m = make_cx<R>(-t.y * o.y, t.y * o.x);
        else m = make_cx<R>(fma_r(t.x, o.x, -(t.y * o.y)), fma_r(t.x, o.y, t.y * o.x));
        o = make_cx<R>(e.x - m.x, e.y - m.y);
        e = make_cx<R>(e.x + m.x, e.y + m.y);
        return;
    }
    const R px = fma_r(-t.y, o.y, fma_r(t.x, o.x, e.x)), py = fma_r(t.y, o.x, fma_r(t.x, o.y, e.y));
    if constexpr (KIND == DIRECT)
        o = make_cx<R>(fma_r(t.y, o.y, fma_r(-t.x, o.x, e.x)), fma_r(-t.y, o.x, fma_r(-t.x, o.y, e.y)));
    else
        o = make_cx<R>(fma_r(R(2), e.x, -px), fma_r(R(2), e.y, -py));
    e = make_cx<R>(px, py);
}

// a * w_32^{-E}
template <int E, typename R>
__device__ __forceinline__ cx<R> mul_w32(cx<R> a)
{
    constexpr R c1 = R(0.98078528040323044912618223613424), s1 = R(0.19509032201612826784828486847702);
    constexpr R c2 = R(PACO_C8), s2 = R(PACO_S8);
    constexpr R c3 = R(0.83146961230254523707878837761791), s3 = R(0.55557023301960222474283081394853);
    constexpr int q = E & 31;
    if constexpr (q == 0) return a;
    else if constexpr (q == 1) return mul_const(a, c1, -s1);
    else if constexpr (q == 2) return mul_const(a, c2, -s2);
    else if constexpr (q == 3) return mul_const(a, c3, -s3);
    else if constexpr (q == 4) return mul_w8_1(a);
    else if constexpr (q == 5) return mul_const(a, s3, -c3);
    else if constexpr (q == 6) return mul_const(a, s2, -c2);
    else if constexpr (q == 7) return mul_const(a, s1, -c1);
    else return mul_mi(mul_w32<q - 8>(a));
}

template <int S, int R_, typename R>
__device__ __forceinline__ void tw32_row(cx<R> *v)
{
    if constexpr (R_ < 8) {
        v[S * 8 + R_] = mul_w32<S * R_>(v[S * 8 + R_]);
        tw32_row<S, R_ + 1>(v);
    }
}

// 32-point DFT: radix 4 over r, r + 8, r + 16, r + 24, twiddle w_32^{-s r},
// radix 8 over r; k = s + 4 m.
template <typename R>
__device__ __forceinline__ void dft32(cx<R> *v)
{
#pragma unroll
    for (int r = 0; r < 8; ++r) dft4_s(v[r], v[r + 8], v[r + 16], v[r + 24]);
    tw32_row<1, 1>(v);
    tw32_row<2, 1>(v);
    tw32_row<3, 1>(v);
    cx<R> y[32];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        dft8(v + 8 * s);
#pragma unroll
        for (int m = 0; m < 8; ++m) y[s + 4 * m] = v[8 * s + m];
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = y[k];
}

// the plain DFT of a pass without twiddles
template <int RADIX, typename R>
__device__ __forceinline__ void plain_dft(cx<R> *v)
{
    if constexpr (RADIX == 32) dft32(v);
    else dft<RADIX>(v);
}

// One level: size n of an RADIX-point DFT held in bit-reversed order in u.
// tau(q) with q = tau_index(n, s) is T^(RADIX / n) w_n^{-s}, s < n / 4 (s = 0 for n = 2, 4).
__host__ __device__ constexpr int tau_index(int n, int s) { return n == 2 ? 0 : n / 4 + s; }

template <int KIND, typename R, int RADIX, int N_, class Tau>
__device__ __forceinline__ void fold_level(cx<R> *u, const Tau &tau)
{
    constexpr int Q = N_ >= 4 ? N_ / 4 : 1;
#pragma unroll
    for (int s = 0; s < Q; ++s) {
        const cx<R> t = tau(tau_index(N_, s));
#pragma unroll
        for (int b = 0; b < RADIX; b += N_) {
            bfly<KIND>(u[b + s], u[b + s + N_ / 2], t);
            if constexpr (N_ >= 4) bfly<KIND>(u[b + s + Q], u[b + s + Q + N_ / 2], make_cx<R>(t.y, -t.x));
        }
    }
    if constexpr (N_ < RADIX) fold_level<KIND, R, RADIX, N_ * 2>(u, tau);
}

template <int RADIX>
__host__ __device__ constexpr int bitrev_c(int i)
{
    int r = 0;
    for (int b = 1; b < RADIX; b <<= 1) r = (r << 1) | ((i & b) ? 1 : 0);
    return r;
}

// v[k] = sum_r v[r] T^r w_RADIX^{-rk}
template <int KIND, typename R, int RADIX, class Tau>
__device__ __forceinline__ void fold_dft(cx<R> *v, const Tau &tau)
{
    cx<R> u[RADIX];
#pragma unroll
    for (int i = 0; i < RADIX; ++i) u[i] = v[bitrev_c<RADIX>(i)];
    fold_level<KIND, R, RADIX, 2>(u, tau);
#pragma unroll
    for (int i = 0; i < RADIX; ++i) v[i] = u[i];
}

// Whether one of N values is so large that a sum of 2^lg of them (a DFT's result, or
// a partial one: at most sqrt(2) 2^lg times the largest part) may overflow.  Every
// tile of CARRY butterflies asks this of its input at its exchange's barrier, and
// is done again with SAFE ones where one thread says yes.
template <int N>
__device__ __forceinline__ bool may_overflow(const cx<float> *v, int lg)
{
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(v[i].x), "f"(v[i].y));
    return m >= __uint_as_float((unsigned)(127 + 126 - lg) << 23);
}
template <int N>
__device__ __forceinline__ bool may_overflow(const cx<double> *v, int lg)
{
    // by the high words: the FP64 pipe is what bounds these passes
    int m = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
        m = max(max(m, __double2hiint(v[i].x) & 0x7fffffff), __double2hiint(v[i].y) & 0x7fffffff);
    return m >= (1023 + 1022 - lg) << 20;
}

// With kappa = 0, F2 is plain and w_L^{-k_lo j_lo} a product of its own in FP64 and
// where F2 is short (at most 8 points: the pass is bound by memory either way,
// and the plain DFT is the closer one), else folded.
__host__ __device__ constexpr bool fold_plain(bool fp64, int lgB) { return fp64 || lgB < 4; }

// EPT_: points a thread holds (0: 16, or 32 where a factor needs them).
// SCALED_: FIRST with FoldArgs::mult and scale (a kernel of its own: with a branch in
// the one kernel 23 x 1024^2 went from 145 to 147 us).
// CLOSER_: F2 in the DIRECT form (FP64 routes of three passes and more).
template <typename R_, int LGA_, int LGB_, int LGW_, bool FIRST_, int TW_, int EPT_ = 0, bool SCALED_ = false,
          bool CLOSER_ = false>
struct FoldCfg {
    using R = R_;
    static constexpr int LGA = LGA_, LGB = LGB_, LGW = LGW_;
    static constexpr bool FIRST = FIRST_, SCALED = SCALED_;
    static constexpr int TW = FIRST_ ? 0 : TW_;
    static constexpr int A = 1 << LGA, B = 1 << LGB, W = 1 << LGW, L = A * B;
    static constexpr int EPT = EPT_ ? EPT_ : A > B ? (A > 16 ? A : 16) : (B > 16 ? B : 16);
    static constexpr int NT = L * W / EPT;
    static constexpr int U1 = EPT / A, U2 = EPT / B;
    // exchange layouts as in paco_power.cuh; PH points make one shared-memory phase
    static constexpr int PH = sizeof(R) == 4 ? 16 : 8;
    static constexpr int SJ = FIRST ? A + 1 : W;
    static constexpr int SC0 = B * SJ;
    static constexpr int SC = FIRST ? SC0 + (((W < PH ? PH / W : 1) - SC0 % PH + PH) % PH) : 1;
    static constexpr int SK = FIRST ? 1 : B * W + (W < PH ? (W - (B * W) % PH + PH) % PH : 0);
    static constexpr int EX = FIRST ? W * SC : A * SK;
    static constexpr bool FP64 = sizeof(R) == 8;
    static constexpr bool PLAIN2 = TW == 0 && fold_plain(FP64, LGB);   // F2 without factors of its own
    // F1's factors read ahead of the tile, with 16 points a thread (2^28 points: 128
    // 0.648 -> 0.610 ms).  With 32 they cost more than they hide: 512 0.66 -> 0.72;
    // 1024 0.853 -> 0.834, but one 2^20 12.3 -> 14.3 us.
    static constexpr bool AHEAD = TW == 1 && !FP64 && EPT == 16;
    static constexpr bool ROWS = TW && FP64;                      // F1's factors by row (T^r), not by level
    // The butterflies of F1 and F2 (bfly): CARRY with may_overflow's question, or DIRECT
    // where that costs less.  us without the question, with it, and with DIRECT: 16 x
    // 2^24 (256 points) 2012, 2013, 2073; 50 x 2^20 (1024 points, TW 1) 326.8, 327.4,
    // 337.9; but 2^28 (512 points, TW 2) 2283, 2385, 2345, and the 2-D form's 1024 points
    // (23 x 1024^2) 144.8, 150.8, 146.4.
    static constexpr int BFLY1 = TW == 2 && EPT == 32 ? DIRECT : CARRY;
    // In FP64 the error decides (relative L2 against a long-double FFT; stage kernels,
    // CARRY, DIRECT): 2^18 2.90e-16, 2.82, -; but 2^20 3.05e-16, 3.08, 2.97, 2^22 3.18,
    // 3.22, 3.12, 2^24 3.32, 3.42, 3.29.  From three passes on (TW 2 among them) F2 is
    // DIRECT: 2^27 21.1 -> 22.5 ms.
    static constexpr int BFLY2 = CLOSER_ || TW == 2 || (TW == 0 && !FP64) ? DIRECT : CARRY;
    static constexpr bool CARRIES = (TW && !ROWS && BFLY1 == CARRY) || (!PLAIN2 && BFLY2 == CARRY);
    static constexpr int NA = ROWS ? A : A / 2;                   // factors of F1, a column
    static constexpr int NTW = TW == 2 ? (NA + LGB) * W : 0;
    static constexpr int SMEM = (EX + NTW) * 2 * (int)sizeof(R);
    static constexpr int REGS = EPT * 2 * (int)sizeof(R) / 4 + (sizeof(R) == 4 ? (EPT == 32 ? 64 : 32) : 64);
    static constexpr int REGS_CTAS = 65536 / (REGS * NT);
    static constexpr int SMEM_CTAS = (227 * 1024) / (SMEM + 1024);
    static constexpr int MINB = REGS_CTAS < 1 ? 1 : (REGS_CTAS < SMEM_CTAS ? REGS_CTAS : SMEM_CTAS);
};

// Programmatic dependent launch: the next kernel of the stream may start its
// CTAs (they read tables only) as this one's last ones run; grid_wait holds
// until the kernels before are complete.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A load of the caller's data (transform, weights, scale) in such a kernel: the
// kernel before may still be writing it when this one starts, so it is neither
// __ldg (the read-only path asks for data that nothing writes as long as the
// kernel runs, its wait included) nor a load that the compiler may move over
// grid_wait (volatile).  Through L2, as the passes run in place.
__device__ __forceinline__ float ld_data(const float *p)
{
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_data(const double *p)
{
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_data(const float2 *p)
{
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_data(const double2 *p)
{
    double2 v;
    asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// One tile of the transform at element offset boff (PDL: the tile's kernel was
// launched with programmatic serialisation).  True: nothing was stored, the tile
// is to be done with AGAIN (may_overflow).
template <class CFG, bool PDL = false, bool AGAIN = false>
__device__ __forceinline__ bool fold_tile(const FoldArgs<typename CFG::R> &a, int tile, long long boff,
                                          unsigned char *smem_raw)
{
    using R = typename CFG::R;
    using C = cx<R>;
    using V = typename vec2<R>::type;
    constexpr int A = CFG::A, B = CFG::B, W = CFG::W, NT = CFG::NT, U1 = CFG::U1, U2 = CFG::U2;
    constexpr bool FIRST = CFG::FIRST;
    constexpr int TW = CFG::TW;
    C *sm = reinterpret_cast<C *>(smem_raw);
    [[maybe_unused]] C *tabA = sm + CFG::EX;       // TW 2: [tau index][col]
    [[maybe_unused]] C *tabB = tabA + CFG::NA * W; //       [i][col]: w_{K L}^{-kappa 2^i}
    const int tid = threadIdx.x;
    const int blk = FIRST ? 0 : tile >> a.lg_tiles;
    const unsigned c0 = (unsigned)(FIRST ? tile : tile & ((1 << a.lg_tiles) - 1)) << CFG::LGW;
    const long long base = boff + (long long)blk * (FIRST ? 0u : a.blk_stride) + c0;

    // TW 2: the columns' factors.  With 32 points a thread their reads go out
    // before the tile's (512 points 0.78 -> 0.75 ms per 2^28); with 16 they would hold
    // up too many small tiles (256: 0.65, 0.68).
    constexpr int NI = (CFG::NTW + NT - 1) / NT;
    [[maybe_unused]] V twl[NI ? NI : 1];
    [[maybe_unused]] auto load_twiddles = [&] {
#pragma unroll
        for (int k = 0; k < NI; ++k) {
            const int e = tid + NT * k;
            if (CFG::NTW % NT == 0 || e < CFG::NTW)
                twl[k] = __ldg(reinterpret_cast<const V *>(a.tau) + CFG::L / 2 + ((unsigned)(e >> CFG::LGW) << a.lg_k) + c0 +
                               (e & (W - 1)));
        }
    };
    if constexpr (TW == 2 && CFG::EPT == 32) load_twiddles();

    [[maybe_unused]] V ahead[CFG::AHEAD ? U1 : 1][CFG::AHEAD ? A / 2 : 1];
    if constexpr (CFG::AHEAD) {
#pragma unroll
        for (int u = 0; u < U1; ++u)
#pragma unroll
            for (int q = 0; q < A / 2; ++q)
                ahead[u][q] = __ldg(reinterpret_cast<const V *>(a.tau) + c0 + ((tid + NT * u) & (W - 1)) + ((unsigned)q << a.lg_k));
    }
    if constexpr (PDL) grid_wait();
    // ---- F1
    [[maybe_unused]] R f = R(1);
    if constexpr (CFG::SCALED) f = a.scale ? a.mult * (R)ld_data(a.scale) : a.mult;
    C v[CFG::EPT];
#pragma unroll
    for (int u = 0; u < U1; ++u) {
        const int s = tid + NT * u, col = s & (W - 1), jlo = s >> CFG::LGW;
        const unsigned jrow = a.rev_bits ? digit_reverse((unsigned)jlo, a.rev_bits, a.rev_t) : (unsigned)jlo;
        const V *p = reinterpret_cast<const V *>(a.in + base + col + (long long)jrow * a.ld_in);
        if (a.conj) {
#pragma unroll
            for (int r = 0; r < A; ++r) {
                const V t = ld_data(p + a.rowA[r]);
                v[u * A + r] = make_cx<R>(t.y, t.x);
            }
        } else {
#pragma unroll
            for (int r = 0; r < A; ++r) {
                const V t = ld_data(p + a.rowA[r]);
                v[u * A + r] = make_cx<R>(t.x, t.y);
            }
        }
    }
    if constexpr (CFG::SCALED) {
        // the input, not the result: a sum may overflow where the scaled one does not
#pragma unroll
        for (int i = 0; i < CFG::EPT; ++i) v[i] = make_cx<R>(v[i].x * f, v[i].y * f);
    }
    [[maybe_unused]] bool again = false;
    if constexpr (CFG::CARRIES && !AGAIN) again = may_overflow<CFG::EPT>(v, CFG::LGA + CFG::LGB);
    if constexpr (AGAIN) __syncthreads();          // the exchange has been read
    if constexpr (TW == 2) {
        if constexpr (CFG::EPT != 32) load_twiddles();
#pragma unroll
        for (int k = 0; k < NI; ++k)
            if (CFG::NTW % NT == 0 || tid + NT * k < CFG::NTW) tabA[tid + NT * k] = make_cx<R>(twl[k].x, twl[k].y);
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < U1; ++u) {
        const int s = tid + NT * u, col = s & (W - 1), jlo = s >> CFG::LGW;
        const V *t1 = reinterpret_cast<const V *>(a.tau);
        C *ex = sm + (FIRST ? col * CFG::SC + jlo * CFG::SJ : jlo * W + col);
        if constexpr (TW == 0) {
            plain_dft<A>(v + u * A);
            if constexpr (CFG::PLAIN2) {
#pragma unroll
                for (int k = 1; k < A; ++k) {
                    const V t = __ldg(t1 + k * jlo);         // w_L^{-k_lo j_lo}
                    v[u * A + k] = cmul(v[u * A + k], make_cx<R>(t.x, t.y));
                }
            }
        } else {
            t1 += c0 + col;
            auto f1 = [&](int q) {
                if constexpr (TW == 2) return tabA[q * W + col];
                if constexpr (CFG::AHEAD) return make_cx<R>(ahead[u][q].x, ahead[u][q].y);
                const V t = __ldg(t1 + ((unsigned)q << a.lg_k));
                return make_cx<R>(t.x, t.y);
            };
            if constexpr (CFG::ROWS) {
#pragma unroll
                for (int r = 1; r < A; ++r) v[u * A + r] = cmul(v[u * A + r], f1(r));
                plain_dft<A>(v + u * A);
            } else {
                fold_dft<AGAIN ? SAFE : CFG::BFLY1, R, A>(v + u * A, f1);
            }
        }
#pragma unroll
        for (int k = 0; k < A; ++k) ex[FIRST ? k : k * CFG::SK] = v[u * A + k];
    }
    // (the answer is asked for after F2, whose table reads would else wait for it)
    if constexpr (CFG::CARRIES && !AGAIN) again = __syncthreads_or(again);
    else __syncthreads();
    // ---- F2
#pragma unroll
    for (int u = 0; u < U2; ++u) {
        const int s = tid + NT * u;
        int col, klo;
        if constexpr (FIRST) { klo = s & (A - 1); col = s >> CFG::LGA; }
        else { col = s & (W - 1); klo = s >> CFG::LGW; }
        const C *ex = sm + (FIRST ? col * CFG::SC + klo : klo * CFG::SK + col);
#pragma unroll
        for (int r = 0; r < B; ++r) v[u * B + r] = ex[r * CFG::SJ];
        if constexpr (CFG::PLAIN2) {
            plain_dft<B>(v + u * B);
        } else {
            // factor q of (k_lo, column): entry q A + k_lo after F1's
            const V *t2 = reinterpret_cast<const V *>(a.tau);
            if constexpr (TW == 1) t2 += c0 + col + ((unsigned)(CFG::NA + klo) << a.lg_k);
            else t2 += klo;
            fold_dft<AGAIN ? SAFE : CFG::BFLY2, R, B>(v + u * B, [&](int q) {
                const V t = __ldg(t2 + (TW == 1 ? (unsigned)(q * A) << a.lg_k : (unsigned)(q * A)));
                const C w = make_cx<R>(t.x, t.y);
                if constexpr (TW != 2) return w;
                int lg = 0;                                  // B / n = 2^lg
                while ((q == 0 ? 2 : 4 << (31 - __clz(q))) << lg < B) ++lg;
                return cmul(w, tabB[lg * W + col]);
            });
        }
        if constexpr (CFG::CARRIES && !AGAIN)
            if (u == 0 && again) return true;
        V *q;
        if constexpr (FIRST) {
            const unsigned c = c0 + col;
            const unsigned row = a.crev_bits ? digit_reverse(c, a.crev_bits, a.crev_t) : c;
            q = reinterpret_cast<V *>(a.out + boff + (long long)row * a.ld_out + klo);
        } else {
            q = reinterpret_cast<V *>(a.out + base + col + (long long)klo * a.ld_out);
        }
        // parts swapped back: at the stores, or (first pass of 512 points) in a branch
        // before them, which keeps the stores behind all of the sequence's F2 (200 x
        // 2^18: 261 us, with selects 273; 301 x 2^16, with a first pass of 256: 97 and 95)
        constexpr bool SWAP = FIRST && CFG::EPT == 32 && U2 > 1;
        if constexpr (SWAP) {
            if (a.conj) {
#pragma unroll
                for (int k = 0; k < B; ++k) v[u * B + k] = make_cx<R>(v[u * B + k].y, v[u * B + k].x);
            }
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const C y = v[u * B + k];
            V o;
            o.x = !SWAP && a.conj ? y.y : y.x;
            o.y = !SWAP && a.conj ? y.x : y.y;
            if constexpr (FIRST) q[A * k] = o;
            else __stcs(q + a.rowK[k], o);
        }
    }
    return false;
}

// The transform's tile and offset of a CTA.  Every second pass takes the tiles
// from the end: what the pass before it wrote last is still in L2.
template <typename R>
__device__ __forceinline__ void fold_cta(const FoldArgs<R> &a, int *tile, long long *boff)
{
    const unsigned b = a.reverse ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
    *tile = (int)(b & ((1u << a.lg_all) - 1u));
    *boff = (long long)(b >> a.lg_all) * a.bstride;
}

// The tile with AGAIN, out of line.
template <class CFG>
__device__ __noinline__ void fold_again(const FoldArgs<typename CFG::R> &a, unsigned char *smem_raw)
{
    int tile;
    long long boff;
    fold_cta(a, &tile, &boff);
    fold_tile<CFG, false, true>(a, tile, boff, smem_raw);
}

template <class CFG>
__global__ void __launch_bounds__(CFG::NT, CFG::MINB) paco_fold_kernel(const __grid_constant__ FoldArgs<typename CFG::R> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_launch_dependents();
    int tile;
    long long boff;
    fold_cta(a, &tile, &boff);
    if (fold_tile<CFG, true>(a, tile, boff, smem_raw)) {
        if constexpr (CFG::CARRIES) {
            // (in line for 256 and 512 points, 16 x 2^24 2013 us for 2057; the others
            // spill for it, one 2^20 10.30 us for 10.01)
            if constexpr (CFG::LGB != 4) {
                fold_again<CFG>(a, smem_raw);
            } else {
                fold_cta(a, &tile, &boff);
                fold_tile<CFG, false, true>(a, tile, boff, smem_raw);
            }
        }
    }
}

// What the host needs to launch one of the kernels above.
struct FoldKernel {
    const void *fn = nullptr;
    int lgA = 0, lgB = 0, lgW = 0, threads = 0, smem = 0;
};

template <class CFG>
FoldKernel fold_kernel_of()
{
    FoldKernel k;
    k.fn = reinterpret_cast<const void *>(&paco_fold_kernel<CFG>);
    k.lgA = CFG::LGA;
    k.lgB = CFG::LGB;
    k.lgW = CFG::LGW;
    k.threads = CFG::NT;
    k.smem = CFG::SMEM;
    return k;
}

// The launch constants of pass i of the n factors f (log2; first pass first),
// tables aside: k.lgA, k.lgB and k.lgW are read.
template <typename R>
void fold_pass_args(FoldArgs<R> *a, const FoldKernel &k, const int *f, int n, int i, int t);

// A device table for FoldArgs::tau in mode FoldCfg::TW, 2^lgK columns.
// kappa = 0 for every column where no_kappa is set.  The first `skip` bytes of
// *dst (a multiple of 16) are left to the caller.
template <typename R>
paco_status_t fold_table(void **dst, const FoldKernel &k, int mode, int lgK, bool no_kappa = false, size_t skip = 0);
// The complex64 table of mode 0 (2^(lgL - 1) factors of F2) at dst.
void fold_levels(void *dst, const FoldKernel &k);

// The kernel for a pass of length 2^lgL whose row blocks have 2^lgC columns
// (the row stride); fn == nullptr where none is built.  scaled: the first pass of a
// scaled input.
FoldKernel fold_kernel_f32(bool first, int tw, int lgL, int lgC, bool narrow, bool scaled = false);
// closer: a later pass of three or more.
FoldKernel fold_kernel_f64(bool first, int tw, int lgL, int lgC, bool closer);

} // namespace paco
