// paco_tcpass.cuh -- a local-FFT pass of a tensor-core precision form whose
// radix-16 sub-DFTs go from memory to mma fragments and back without staging.
//
// The contraction is that of paco_tc.cuh ([Re y; Im y] = M [Re x; Im x], mma
// m16n8k16, the same terms and the same order of products).  There a lane holds
// a whole sequence and the operands pass through shared memory on both sides;
// here the lane (g, q) of a warp loads exactly what the B fragment wants of it,
// points 2q, 2q+1, 2q+8, 2q+9 of sequence g, and keeps what the accumulators
// give it, frequencies g and g + 8 of sequences 2q and 2q + 1, so that the
// twiddle and the exchange (or the result's store) follow from the fragments.
// The stage kernels spent 180 instructions a point on two contractions, 110 of
// them on run-time strides: 6 x 2^22 BF16x3 took 669 us, and takes 359.
//
// Layout of a pass as in paco_fold.cuh: L = 16 B rows, j = j_hi B + j_lo, k =
// k_lo + 16 k_hi, a tile of W columns, FIRST with the redistribution in its
// stores, else in place with w_{K L}^{-kappa j} (kappa = column) multiplied into
// the input.  F1 is a contraction; F2 is one too (TC2, B = 16) or a plain
// B-point DFT.  A route has at most four contractions, as the stage kernels had:
// each adds its truncating accumulation to the error.
//
// Exchange (in points): FIRST [col][j_lo][k_lo], else [k_lo][j_lo][col], rows of
// 16 or W places padded by two: fragment reads (4 sequences x 4 rows a
// half-warp) and the writes (8 or 16 bytes) hit every bank once.
#pragma once

#include "paco_fold.cuh"
#include "paco_tc.cuh"

namespace paco {

struct TcPassArgs {
    FoldArgs<float> f;      // strides, row maps (rowK aside)
    const cx<float> *twL;   // w_L^{-r}, r < L
    const cx<float> *lo;    // w_N^{-r}, r < 2^lo_bits
    const cx<float> *hi;    // w_N^{-(r << lo_bits)}
    int lo_bits;
    const uint4 *frag;      // the matrix fragments (tc_table_create)
};

// The contraction of 32 sequences in fragment distribution: x[nt][i] is point
// 2q + (i & 1) + 8 (i >> 1) of sequence 8 nt + g; y[nt][si][h] becomes frequency
// g + 8 si of sequence 8 nt + 2q + h.
template <int FORM>
__device__ __forceinline__ void tc_fragments(const cx<float> (&x)[4][4], const uint4 *tab, cx<float> (&y)[4][2][2])
{
    using T = TcForm<FORM>;
    const int lane = threadIdx.x & 31, q = lane & 3;
    float acc[4][2][4];
    float sc[4], back[4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) acc[nt][mt][0] = acc[nt][mt][1] = acc[nt][mt][2] = acc[nt][mt][3] = 0.f;
        sc[nt] = back[nt] = 1.f;
        if constexpr (FORM == TC_FP16) {
            // the sequence's scale, its largest component in [1, 2) (four lanes hold it)
            float mx = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) mx = fmaxf(mx, fmaxf(fabsf(x[nt][i].x), fabsf(x[nt][i].y)));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            int e = (int)((__float_as_uint(mx) >> 23) & 0xff) - 127;
            if (e < -100) e = -100;
            if (e > 100) e = 100;
            sc[nt] = __uint_as_float((uint32_t)(127 - e) << 23);
            back[nt] = __uint_as_float((uint32_t)(127 + e) << 23);
        }
    }
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {                      // Re x, Im x
        uint4 af[2][T::TA];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int ta = 0; ta < T::TA; ++ta) af[mt][ta] = tab[((ta * 2 + mt) * 2 + ks) * 32 + lane];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            float r[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = ks ? x[nt][i].y : x[nt][i].x;
            uint32_t b[T::TB][2];
            if constexpr (FORM == TC_BF16X3) {
#pragma unroll
                for (int t = 0; t < 3; ++t)
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        const __nv_bfloat162 h = __floats2bfloat162_rn(r[2 * w], r[2 * w + 1]);
                        b[t][w] = *reinterpret_cast<const uint32_t *>(&h);
                        if (t < 2) {
                            const float2 hf = __bfloat1622float2(h);
                            r[2 * w] -= hf.x;
                            r[2 * w + 1] -= hf.y;
                        }
                    }
            } else {
                b[0][0] = pack_f16(r[0] * sc[nt], r[1] * sc[nt]);
                b[0][1] = pack_f16(r[2] * sc[nt], r[3] * sc[nt]);
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float *d = acc[nt][mt];
                if constexpr (FORM == TC_BF16X3) {        // smallest products first
                    mma_bf16(d, af[mt][2], b[0][0], b[0][1]);
                    mma_bf16(d, af[mt][1], b[1][0], b[1][1]);
                    mma_bf16(d, af[mt][0], b[2][0], b[2][1]);
                    mma_bf16(d, af[mt][1], b[0][0], b[0][1]);
                    mma_bf16(d, af[mt][0], b[1][0], b[1][1]);
                    mma_bf16(d, af[mt][0], b[0][0], b[0][1]);
                } else {
                    mma_f16(d, af[mt][1], b[0][0], b[0][1]);
                    mma_f16(d, af[mt][0], b[0][0], b[0][1]);
                }
            }
        }
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s = 1.f;
            if constexpr (FORM == TC_FP16) s = __shfl_sync(0xffffffffu, back[nt], 4 * (2 * q + h));
#pragma unroll
            for (int si = 0; si < 2; ++si)
                y[nt][si][h] = make_cx<float>(acc[nt][0][h + 2 * si] * s, acc[nt][1][h + 2 * si] * s);
        }
}

template <int FORM_, int LGB_, int LGW_, bool FIRST_, bool TC2_>
struct TcPassCfg {
    static constexpr int FORM = FORM_, LGB = LGB_, LGW = LGW_;
    static constexpr bool FIRST = FIRST_, TC2 = TC2_;
    static constexpr int A = 16, B = 1 << LGB, W = 1 << LGW, L = A * B, NT = B * W;
    static_assert(!TC2 || B == 16, "a contraction is 16 points");
    static_assert(W >= 8 && NT % 32 == 0, "eight columns a fragment");
    static constexpr int SJ = (FIRST ? A : W) + 2;
    static constexpr int SC = FIRST ? B * SJ + 2 : 1;              // FIRST: points of a column
    static constexpr int SK = FIRST ? 1 : (B * SJ + 7) / 16 * 16 + 8;   // else: points of a k_lo
    static constexpr int EX = FIRST ? W * SC : A * SK;
    static constexpr int NTW = FIRST ? 0 : (A + B) * W;            // the columns' input factors
    static constexpr int SMEM = TcForm<FORM>::TABLE_U4 * 16 + (EX + NTW) * 8;
    static constexpr int CTAS = 512 / NT < (227 * 1024) / (SMEM + 1024) ? 512 / NT : (227 * 1024) / (SMEM + 1024);
};

template <class CFG>
__global__ void __launch_bounds__(CFG::NT, CFG::CTAS) paco_tcpass_kernel(const __grid_constant__ TcPassArgs args)
{
    using C = cx<float>;
    constexpr int A = CFG::A, B = CFG::B, W = CFG::W, NT = CFG::NT, LGW = CFG::LGW;
    constexpr bool FIRST = CFG::FIRST;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint4 *tab = reinterpret_cast<uint4 *>(smem_raw);
    C *sm = reinterpret_cast<C *>(tab + TcForm<CFG::FORM>::TABLE_U4);
    [[maybe_unused]] C *rows = sm + CFG::EX;       // [j_hi][col]: w_{16 K}^{-kappa j_hi}
    [[maybe_unused]] C *cols = rows + A * W;       // [j_lo][col]: w_{K L}^{-kappa j_lo}
    const FoldArgs<float> &a = args.f;
    const int tid = threadIdx.x, lane = tid & 31, w0 = tid & ~31, g = lane >> 2, q = lane & 3;
    grid_launch_dependents();
    const unsigned bid = a.reverse ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
    const int tile = (int)(bid & ((1u << a.lg_all) - 1u));
    const long long boff = (long long)(bid >> a.lg_all) * a.bstride;
    const int blk = FIRST ? 0 : tile >> a.lg_tiles;
    const unsigned c0 = (unsigned)(FIRST ? tile : tile & ((1 << a.lg_tiles) - 1)) << LGW;
    const long long base = boff + (long long)blk * (FIRST ? 0u : a.blk_stride) + c0;

    for (int r = tid; r < TcForm<CFG::FORM>::TABLE_U4; r += NT) tab[r] = __ldg(args.frag + r);
    // the columns' factors: their table reads go out before the tile's
    constexpr int NI = (CFG::NTW + NT - 1) / NT;
    [[maybe_unused]] float2 tl[NI ? NI : 1], th[NI ? NI : 1];
    if constexpr (!FIRST) {
        const int lgL = 4 + CFG::LGB, sh = a.lg_n - a.lg_k;        // w_{K M} = w_N^(N / (K M))
#pragma unroll
        for (int k = 0; k < NI; ++k) {
            const int e = tid + NT * k, r = e >> LGW;
            const unsigned kap = c0 + (e & (W - 1));
            const unsigned ex = r < A ? (kap * (unsigned)r) << (sh - 4) : (kap * (unsigned)(r - A)) << (sh - lgL);
            if (CFG::NTW % NT == 0 || e < CFG::NTW) {
                tl[k] = __ldg(reinterpret_cast<const float2 *>(args.lo + (ex & ((1u << args.lo_bits) - 1u))));
                th[k] = __ldg(reinterpret_cast<const float2 *>(args.hi + (ex >> args.lo_bits)));
            }
        }
    }
    grid_wait();
    // ---- F1: the fragments of this warp's 32 sequences, straight from memory
    C x[4][4];
    const unsigned rq = ((q & 1) ? a.rowA[2] : 0u) + ((q & 2) ? a.rowA[4] : 0u);   // (row maps are linear in bits)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int s = w0 + 8 * nt + g, col = s & (W - 1), jlo = s >> LGW;
        const unsigned jrow = a.rev_bits ? digit_reverse((unsigned)jlo, a.rev_bits, a.rev_t) : (unsigned)jlo;
        const float2 *p = reinterpret_cast<const float2 *>(a.in + base + col + (long long)jrow * a.ld_in) + rq;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 t = ld_data(p + ((i & 1) ? a.rowA[1] : 0u) + ((i & 2) ? a.rowA[8] : 0u));
            x[nt][i] = a.conj ? make_cx<float>(t.y, t.x) : make_cx<float>(t.x, t.y);
        }
    }
    if constexpr (!FIRST) {
#pragma unroll
        for (int k = 0; k < NI; ++k)
            if (CFG::NTW % NT == 0 || tid + NT * k < CFG::NTW)
                rows[tid + NT * k] = cmul(make_cx<float>(tl[k].x, tl[k].y), make_cx<float>(th[k].x, th[k].y));
    }
    __syncthreads();
    if constexpr (!FIRST) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int s = w0 + 8 * nt + g, col = s & (W - 1), jlo = s >> LGW;
            const C gc = cols[jlo * W + col];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x[nt][i] = cmul(x[nt][i], cmul(gc, rows[(2 * q + (i & 1) + 8 * (i >> 1)) * W + col]));
        }
    }
    C y[4][2][2];
    tc_fragments<CFG::FORM>(x, tab, y);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int s = w0 + 8 * nt + 2 * q, col = s & (W - 1), jlo = s >> LGW;   // and column + 1
#pragma unroll
        for (int si = 0; si < 2; ++si) {
            const int klo = g + 8 * si;
            const float2 t = __ldg(reinterpret_cast<const float2 *>(args.twL) + klo * jlo);
            const C w = make_cx<float>(t.x, t.y);
            const C y0 = cmul(y[nt][si][0], w), y1 = cmul(y[nt][si][1], w);
            if constexpr (FIRST) {
                sm[col * CFG::SC + jlo * CFG::SJ + klo] = y0;
                sm[(col + 1) * CFG::SC + jlo * CFG::SJ + klo] = y1;
            } else {
                *reinterpret_cast<float4 *>(sm + klo * CFG::SK + jlo * CFG::SJ + col) = make_float4(y0.x, y0.y, y1.x, y1.y);
            }
        }
    }
    __syncthreads();
    // ---- F2
    if constexpr (CFG::TC2) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int s = w0 + 8 * nt + g;
            const C *ex = FIRST ? sm + (s >> 4) * CFG::SC + (s & 15) : sm + (s >> LGW) * CFG::SK + (s & (W - 1));
#pragma unroll
            for (int i = 0; i < 4; ++i) x[nt][i] = ex[(2 * q + (i & 1) + 8 * (i >> 1)) * CFG::SJ];
        }
        tc_fragments<CFG::FORM>(x, tab, y);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int s = w0 + 8 * nt + 2 * q;                 // and s + 1: the next k_lo (FIRST) or column
            float2 *p;
            if constexpr (FIRST) {
                const unsigned c = c0 + (unsigned)(s >> 4);
                const unsigned row = a.crev_bits ? digit_reverse(c, a.crev_bits, a.crev_t) : c;
                p = reinterpret_cast<float2 *>(a.out + boff + (long long)row * a.ld_out + (s & 15) + 16 * g);
            } else {
                p = reinterpret_cast<float2 *>(a.out + base + (s & (W - 1)) + (long long)((s >> LGW) + 16 * g) * a.ld_out);
            }
#pragma unroll
            for (int si = 0; si < 2; ++si) {
                const C u = y[nt][si][0], v = y[nt][si][1];
                const float4 o = a.conj ? make_float4(u.y, u.x, v.y, v.x) : make_float4(u.x, u.y, v.x, v.y);
                *reinterpret_cast<float4 *>(p + (FIRST ? 128u : (unsigned)(128u * a.ld_out)) * si) = o;
            }
        }
    } else {
        constexpr int U = 16 / B;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = tid + NT * u;
            int col, klo;
            if constexpr (FIRST) { klo = s & 15; col = s >> 4; }
            else { col = s & (W - 1); klo = s >> LGW; }
            const C *ex = sm + (FIRST ? col * CFG::SC + klo : klo * CFG::SK + col);
            C v[B];
#pragma unroll
            for (int r = 0; r < B; ++r) v[r] = ex[r * CFG::SJ];
            plain_dft<B>(v);
            float2 *p;
            if constexpr (FIRST) {
                const unsigned c = c0 + (unsigned)col;
                const unsigned row = a.crev_bits ? digit_reverse(c, a.crev_bits, a.crev_t) : c;
                p = reinterpret_cast<float2 *>(a.out + boff + (long long)row * a.ld_out + klo);
            } else {
                p = reinterpret_cast<float2 *>(a.out + base + col + (long long)klo * a.ld_out);
            }
#pragma unroll
            for (int k = 0; k < B; ++k)
                p[FIRST ? 16u * k : a.rowK[k]] = a.conj ? make_float2(v[k].y, v[k].x) : make_float2(v[k].x, v[k].y);
        }
    }
}

// The kernel for a pass of length 2^lgL (5..8; FIRST 6..8) whose row blocks
// have 2^lgC columns; fn == nullptr where none is built.
FoldKernel tcpass_kernel(int form, bool first, bool tc2, int lgL, int lgC);

} // namespace paco
