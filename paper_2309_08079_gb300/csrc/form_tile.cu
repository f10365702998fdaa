// Fused formation of S+, gamma and Phi^-1 (Sec. II-B, Sec. IV-A) for the two
// measured float32 shapes: nx = 14, nu = 7 (diagonal or dense costs) and nx =
// 36, nu = 12 (diagonal).  Other shapes, float64 and unaligned arrays take the
// kernels of form.cu; the formulas, and the order of every sum, are theirs.
//
// What bounds it: a knot takes ~10k (nx = 14) or ~200k (nx = 36) multiply-adds
// on 3.2 or 26 KB of inputs and outputs, so with one operand per multiply-add
// from shared memory (row or element per lane) the shared-memory pipe, at 32
// words per clock, is the limit.  Each lane therefore computes a tile of 4
// rows x TC columns (TC = 4: 16 lanes and half a warp per knot; TC = 12: 27
// lanes and a warp per knot) from 16-byte loads, 1/8 or 1/12 load per
// multiply-add.  A lane's rows are GR apart (ti, ti + GR, ...), which puts the
// lanes of one load on different banks at row strides of 20 and 36 words.
// The inversion keeps its tile in registers: each Gauss-Jordan step passes
// the pivot row and column through shared memory.
//
// A CTA takes `kpb` consecutive knots, one group of lanes each, and one more
// group for the knot after the last (formed and inverted, not written), so
// that every Po[k] = -Pd[k+1] So[k] Pd[k] is formed from shared memory.
//
// Measured (GB300, ragged batches of 256): nx = 14, 69,600 knots 151 us against
// 315 with a warp per knot and one operand load per multiply-add; nx = 36,
// 41,000 knots 946 us against 5,200 in five launches (form, inverse, off-
// diagonal, two packings).  ncu: 68 and 65 % of the shared-memory pipe; DRAM
// would allow 45 and 160 us.  The loops over the summation index and over the
// pivots are rolled at nx = 36: fully unrolled, instruction fetch was the
// largest stall (1,490 against 1,825 us at that step).  5 + 1 warps in two
// CTAs per SM instead of 11 + 1 in one: the same time.
// Dense costs (three more inversions a knot by the same elimination): formation
// and recovery of 32 instances, 4,600 knots, 51 us against 224 in four launches.
#include <algorithm>
#include <cstdint>

#include "launch.cuh"

namespace mpcg {

namespace {

template <int NX, int NU>
struct FT {
    static constexpr int TR = 4, TC = NX <= 16 ? 4 : 12;
    static constexpr int GR = (NX + TR - 1) / TR, GC = (NX + TC - 1) / TC;
    static constexpr bool SQUARE = GR == GC && TR == TC;
    static constexpr int GL = GR * GC <= 16 ? 16 : 32;  // lanes per knot
    static constexpr int LD = NX <= 16 ? 20 : NX;       // row stride (words): GR rows on distinct banks
    static constexpr int LB = (NU + 3) / 4 * 4;         // row stride of B
    static constexpr int MAT = NX * LD;
    static constexpr int NP = (NX + 3) / 4 * 4;         // padded vector
    static constexpr int ROWB = GC * TC, COLB = GR * TR;
    // words per knot: X (A, then Pd), Y (A Q^-1), W (B and B R^-1, then D,
    // then A Q^-1 Pd, then Po), the pivot row and column (two parities), six vectors
    // (the two knots of a warp start 16 banks apart)
    static constexpr int USED = 3 * MAT + 2 * (ROWB + COLB) + 6 * NP;
    static constexpr int WORDS = GL == 16 ? (USED - 16 + 31) / 32 * 32 + 16 : USED;
    static constexpr int QWORDS = (MAT + 31) / 32 * 32;  // dense costs: one more block
    static_assert(2 * NX * LB <= MAT, "B and B R^-1 share W");
    // knots per CTA, and CTAs per SM that the registers are held to: 16 half
    // warps, or 12 warps of 17 KB
    static constexpr int KPB_MAX = NX <= 16 ? 15 : 11;
    static constexpr int PER_SM = NX <= 16 ? 3 : 1;
    static constexpr int NTRI = NX * (NX + 1) / 2, NPK = (NTRI + 3) / 4 * 4;  // packed_len(NX)
    static constexpr int VW = NX % 4 == 0 ? 4 : 2;      // words per global access of a block
};

__device__ __forceinline__ bool weight_ok(float v) { return v > 0.f && v <= 3.402823466e38f; }

template <int VW> struct Vw;
template <> struct Vw<2> { using type = float2; };
template <> struct Vw<4> { using type = float4; };

// A block between global memory (dense) and shared memory (row stride LDS_).
template <int R, int Cn, int LDS_, int VW, int GL>
__device__ __forceinline__ void block_out(float *g, const float *s, int t, float sign = 1.f) {
    using V = typename Vw<VW>::type;
    constexpr int PER = Cn / VW;
#pragma unroll
    for (int e0 = 0; e0 < R * PER; e0 += GL) {
        const int e = e0 + t;
        if (e < R * PER) {
            V v = *reinterpret_cast<const V *>(s + (e / PER) * LDS_ + (e % PER) * VW);
            if (sign < 0.f) {
                v.x = -v.x;
                v.y = -v.y;
                if constexpr (VW == 4) {
                    v.z = -v.z;
                    v.w = -v.w;
                }
            }
            *reinterpret_cast<V *>(g + (size_t)e * VW) = v;
        }
    }
}

// Gauss-Jordan inversion without pivoting of an N x N block (N <= NX of the
// layout F) held as register tiles, rows ti + GR r, columns tj + GC c.  Step p
// passes row p and column p through shared memory (two parities, one warp
// barrier).  p = GC c + x: the tile's row and column of the pivot are fixed by
// c alone, so only c is unrolled.  True if a pivot was not positive and finite.
template <class F, int N>
__device__ __forceinline__ bool gj_tile(float (&M)[F::TR][F::TC], float *rowb, float *colb, int tr, int tcb) {
    constexpr int TR = F::TR, TC = F::TC, GC = F::GC, RC = F::GR / F::GC;
    static_assert(F::GR % F::GC == 0, "one tile row per GR / GC tile columns");
    bool bad = false;
#pragma unroll
    for (int pc = 0; pc < (N + GC - 1) / GC; ++pc) {
        const int pr = pc / RC;  // tile row of these pivots
#pragma unroll 1
        for (int x = 0; x < GC; ++x) {
            const int pv = GC * pc + x;
            if (N % GC != 0 && pv >= N) break;
            float *rb = rowb + (pv & 1) * F::ROWB, *cb = colb + (pv & 1) * F::COLB;
            const bool own_row = tr == GC * (pc % RC) + x, own_col = tcb == x;
            if (own_row) {
#pragma unroll
                for (int c = 0; c < TC; c += 4)
                    *reinterpret_cast<float4 *>(rb + tcb * TC + c) = make_float4(M[pr][c], M[pr][c + 1], M[pr][c + 2], M[pr][c + 3]);
            }
            if (own_col)
                *reinterpret_cast<float4 *>(cb + tr * TR) = make_float4(M[0][pc], M[1][pc], M[2][pc], M[3][pc]);
            __syncwarp();
            const float piv_v = rb[x * TC + pc], d = 1.f / piv_v;
            bad |= !weight_ok(piv_v);
            const float4 col4 = *reinterpret_cast<const float4 *>(cb + tr * TR);
            const float col[TR] = {col4.x, col4.y, col4.z, col4.w};
            float row[TC];
#pragma unroll
            for (int c = 0; c < TC; c += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(rb + tcb * TC + c);
                row[c] = v.x * d;
                row[c + 1] = v.y * d;
                row[c + 2] = v.z * d;
                row[c + 3] = v.w * d;
            }
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                const bool piv = r == pr && own_row;
#pragma unroll
                for (int c = 0; c < TC; ++c) {
                    const float u = __fmaf_rn(-col[r], row[c], M[r][c]);
                    M[r][c] = piv ? row[c] : u;
                }
                if (own_col) M[r][pc] = piv ? d : -col[r] * d;
            }
        }
    }
    __syncwarp();  // the buffers may be used again
    return bad;
}

// M <- (M + M^T) / 2 on a square grid: the mirrored entry of M[r][c] sits in
// lane `mirror` as M[c][r].
template <class F>
__device__ __forceinline__ void sym_tile(float (&M)[F::TR][F::TC], int mirror) {
#pragma unroll
    for (int r = 0; r < F::TR; ++r)
#pragma unroll
        for (int c = r; c < F::TC; ++c) {
            const float o1 = __shfl_sync(0xffffffffu, M[r][c], mirror);
            if (c > r) {
                const float o2 = __shfl_sync(0xffffffffu, M[c][r], mirror);
                M[r][c] = 0.5f * (M[r][c] + o2);
                M[c][r] = 0.5f * (M[c][r] + o1);
            } else {
                M[r][r] = 0.5f * (M[r][r] + o1);
            }
        }
}

}  // namespace

template <int NX, int NU, bool DENSE>
__global__ void __launch_bounds__(FT<NX, NU>::GL *(FT<NX, NU>::KPB_MAX + 1), DENSE ? 2 : FT<NX, NU>::PER_SM)
form_tile_kernel(const SchurArgs<float> a, float *Pd, float *Po, float *Sdp, float *Pdp, int kpb) {
    using F = FT<NX, NU>;
    constexpr int TR = F::TR, TC = F::TC, GR = F::GR, GC = F::GC, GL = F::GL, LD = F::LD, LB = F::LB;
    extern __shared__ __align__(16) float sm[];
    const int grp = threadIdx.x / GL, t = threadIdx.x % GL;
    const int ti = t / GC, tj = t % GC;
    const bool tile = t < GR * GC;  // lanes past the grid repeat the last tile and store nothing
    const int tr = tile ? ti : GR - 1, tcb = tile ? tj : GC - 1;
    constexpr int WORDS = F::WORDS + (DENSE ? F::QWORDS : 0);
    float *X = sm + (size_t)WORDS * grp;
    float *Y = X + F::MAT, *D = Y + F::MAT, *Bm = D, *Bs = Bm + NX * LB;
    float *rowb = D + F::MAT, *colb = rowb + 2 * F::ROWB;
    float *iq0 = colb + 2 * F::COLB, *qs = iq0 + F::NP, *iq1 = qs + F::NP, *q1 = iq1 + F::NP, *ir = q1 + F::NP,
          *rs = ir + F::NP;
    float *Qb = X + F::WORDS;  // DENSE: the inverse cost blocks, one after another
    const int kg = blockIdx.x * kpb + grp, total = a.bv.total();
    if ((int)blockIdx.x * kpb >= total) return;  // the grid covers B x N knots, a ragged batch has fewer
    const bool extra = grp == kpb;
    const int kc = min(kg, total - 1);  // groups past the end repeat the last knot and store nothing
    int b = a.bv.owner(kc), k0, Nb;
    a.bv.range(b, k0, Nb);
    const int k = kc - k0;
    const bool mine = kg < total && !extra && grp < kpb;
    const bool first = k == 0;
    const int j = kc - b - 1;  // control index of (A, B, Rd, r, So) for this row (k > 0)
    bool bad = false;

    // nx = 36: where packed entry p (column by column) sits in a block
    __shared__ unsigned short tri[NX == 36 ? F::NTRI : 1];
    if constexpr (NX == 36)
        if (threadIdx.x < NX)
            for (int i = 0; i <= (int)threadIdx.x; ++i) tri[threadIdx.x * (threadIdx.x + 1) / 2 + i] = (unsigned short)(threadIdx.x * LD + i);
    auto pack_out = [&](float *g, const float *m) {
        for (int e = 4 * t; e < F::NPK; e += 4 * GL) {
            float v[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) v[x] = e + x < F::NTRI ? m[tri[min(e + x, F::NTRI - 1)]] : 0.f;
            *reinterpret_cast<float4 *>(g + (size_t)kc * F::NPK + e) = make_float4(v[0], v[1], v[2], v[3]);
        }
    };

    // ---- inputs; the first block row has no A, B -------------------------------
#pragma unroll
    for (int i0 = 0; i0 < NX; i0 += GL) {
        const int i = i0 + t;
        if (i < NX) {
            q1[i] = a.q[(size_t)kc * NX + i];
            float w = 1.f, qv = first ? 0.f : a.q[(size_t)(kc - 1) * NX + i];
            if constexpr (!DENSE) {
                const float v = a.Qd[(size_t)kc * NX + i];
                bad |= !weight_ok(v);
                iq1[i] = 1.f / v;
                if (!first) {
                    w = a.Qd[(size_t)(kc - 1) * NX + i];
                    bad |= !weight_ok(w);
                }
            }
            iq0[i] = 1.f / w;
            qs[i] = qv / w;
        }
    }
    if (t < NU) {
        float v = 1.f, rv = 0.f;
        if (!first) {
            rv = a.r[(size_t)j * NU + t];
            if constexpr (!DENSE) {
                v = a.Rd[(size_t)j * NU + t];
                bad |= !weight_ok(v);
            }
        }
        ir[t] = 1.f / v;
        rs[t] = rv / v;
    }
    if constexpr (NX == 36) __syncthreads();  // tri
    else __syncwarp();
    {
        using V = typename Vw<F::VW>::type;
        constexpr int VW = F::VW, PER = NX / VW;
        const V *Ak = reinterpret_cast<const V *>(a.A + (first ? 0 : (size_t)j * NX * NX));
#pragma unroll
        for (int e0 = 0; e0 < NX * PER; e0 += GL) {
            const int e = e0 + t;
            if (e < NX * PER) {
                V v{};
                if (!first) v = Ak[e];
                const int i = e / PER, c = (e % PER) * VW;
                const V w = *reinterpret_cast<const V *>(iq0 + c);
                V s;
                s.x = v.x * w.x;
                s.y = v.y * w.y;
                if constexpr (VW == 4) {
                    s.z = v.z * w.z;
                    s.w = v.w * w.w;
                }
                *reinterpret_cast<V *>(X + i * LD + c) = v;
                *reinterpret_cast<V *>(Y + i * LD + c) = s;
            }
        }
        const float *Bk = a.B + (first ? 0 : (size_t)j * NX * NU);
#pragma unroll
        for (int e0 = 0; e0 < NX * NU; e0 += GL) {
            const int e = e0 + t;
            if (e < NX * NU) {
                const float v = first ? 0.f : Bk[e];
                Bm[(e / NU) * LB + e % NU] = v;
                Bs[(e / NU) * LB + e % NU] = v * ir[e % NU];
            }
        }
    }
    __syncwarp();

    float M[TR][TC];
    // a tile with strided columns to a block in shared memory
    auto put_strided = [&](float *S, const float (&v)[TR][TC]) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c)
                if (tile && ti + GR * r < NX && tj + GC * c < NX) S[(ti + GR * r) * LD + tj + GC * c] = v[r][c];
    };
    const int mirror = (threadIdx.x & 31 & ~(GL - 1)) + tj * GC + ti;  // the lane of the mirrored tile (square grids)

    float acc[TR][TC];
    auto nn = [&](const float *P, const float *Q, float sign) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) acc[r][c] = 0.f;
#pragma unroll NX % 4 ? 4 : 1
        for (int m = 0; m < NX; m += 4) {
            float x[TR][4];
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                const float4 v = *reinterpret_cast<const float4 *>(P + min(tr + GR * r, NX - 1) * LD + m);
                x[r][0] = sign * v.x;
                x[r][1] = sign * v.y;
                x[r][2] = sign * v.z;
                x[r][3] = sign * v.w;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                if (NX % 4 && m + kk >= NX) continue;
#pragma unroll
                for (int c = 0; c < TC; c += 4) {
                    const float4 y = *reinterpret_cast<const float4 *>(Q + (m + kk) * LD + tcb * TC + c);
#pragma unroll
                    for (int r = 0; r < TR; ++r) {
                        acc[r][c] = __fmaf_rn(x[r][kk], y.x, acc[r][c]);
                        acc[r][c + 1] = __fmaf_rn(x[r][kk], y.y, acc[r][c + 1]);
                        acc[r][c + 2] = __fmaf_rn(x[r][kk], y.z, acc[r][c + 2]);
                        acc[r][c + 3] = __fmaf_rn(x[r][kk], y.w, acc[r][c + 3]);
                    }
                }
            }
        }
    };
    auto put = [&](float *T, float sign) {
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            const int i = ti + GR * r;
            if (tile && i < NX)
#pragma unroll
                for (int c = 0; c < TC; c += 4)
                    *reinterpret_cast<float4 *>(T + i * LD + tj * TC + c) =
                        make_float4(sign * acc[r][c], sign * acc[r][c + 1], sign * acc[r][c + 2], sign * acc[r][c + 3]);
        }
    };

    // ---- dense costs: Q_{k-1}^-1, R_{k-1}^-1 and Q_k^-1 by the same elimination; Y = A
    // Q_{k-1}^-1, Bs = B R_{k-1}^-1; Q_k^-1 stays in M (theta starts from it) and Qb ----
    if constexpr (DENSE) {
        static_assert(F::SQUARE, "dense costs: the square grid");
        // n x n block in global memory to tiles (identity where there is none)
        auto load_tile = [&](const float *g, int n, bool on) {
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int c = 0; c < TC; ++c) {
                    const int i = ti + GR * r, jj = tj + GC * c;
                    M[r][c] = on && i < n && jj < n ? g[i * n + jj] : (i == jj ? 1.f : 0.f);
                }
        };
        load_tile(a.Qf + (first ? 0 : (size_t)(kc - 1) * NX * NX), NX, !first);
        bad |= gj_tile<F, NX>(M, rowb, colb, tr, tcb);
        sym_tile<F>(M, mirror);
        put_strided(Qb, M);
        __syncwarp();
        nn(X, Qb, 1.f);
        put(Y, 1.f);
        __syncwarp();
        load_tile(a.Rf + (first ? 0 : (size_t)j * NU * NU), NU, !first);
        bad |= gj_tile<F, NU>(M, rowb, colb, tr, tcb);
        sym_tile<F>(M, mirror);
        put_strided(Qb, M);
        __syncwarp();
#pragma unroll
        for (int e0 = 0; e0 < NX * NU; e0 += GL) {
            const int e = e0 + t;
            if (e < NX * NU) {
                float v = 0.f;
#pragma unroll
                for (int m = 0; m < NU; ++m) v = __fmaf_rn(Bm[(e / NU) * LB + m], Qb[m * LD + e % NU], v);
                Bs[(e / NU) * LB + e % NU] = v;
            }
        }
        __syncwarp();
        load_tile(a.Qf + (size_t)kc * NX * NX, NX, true);
        bad |= gj_tile<F, NX>(M, rowb, colb, tr, tcb);
        sym_tile<F>(M, mirror);
        put_strided(Qb, M);
        __syncwarp();
    }

    // ---- theta: rows ti + GR r, columns tj + GC c; the upper triangle, mirrored ----
    {
        float acc[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) acc[r][c] = DENSE ? M[r][c] : 0.f;
        auto nt = [&](const float *P, const float *Q, int ld, int m0, int n) {
            float4 x[TR];
#pragma unroll
            for (int r = 0; r < TR; ++r) x[r] = *reinterpret_cast<const float4 *>(P + min(tr + GR * r, NX - 1) * ld + m0);
#pragma unroll
            for (int c = 0; c < TC; ++c) {
                const float4 y = *reinterpret_cast<const float4 *>(Q + min(tcb + GC * c, NX - 1) * ld + m0);
#pragma unroll
                for (int r = 0; r < TR; ++r) {
                    if (F::SQUARE && r > c) continue;  // below the diagonal: mirrored
                    if (n > 0) acc[r][c] = __fmaf_rn(x[r].x, y.x, acc[r][c]);
                    if (n > 1) acc[r][c] = __fmaf_rn(x[r].y, y.y, acc[r][c]);
                    if (n > 2) acc[r][c] = __fmaf_rn(x[r].z, y.z, acc[r][c]);
                    if (n > 3) acc[r][c] = __fmaf_rn(x[r].w, y.w, acc[r][c]);
                }
            }
        };
        // (rolled where every chunk is full: the unrolled products do not fit
        // the instruction cache)
#pragma unroll NX % 4 ? 4 : 1
        for (int m = 0; m < NX; m += 4) nt(Y, X, LD, m, NX % 4 ? NX - m : 4);
#pragma unroll NU % 4 ? 2 : 1
        for (int m = 0; m < NU; m += 4) nt(Bs, Bm, LB, m, NU % 4 ? NU - m : 4);
        // ---- gamma -----------------------------------------------------------------
#pragma unroll
        for (int i0 = 0; i0 < NX; i0 += GL) {
            const int i = i0 + t;
            if (i < NX && mine) {
                const float cv = a.c[(size_t)kc * NX + i];
                float z = DENSE ? 0.f : __fmul_rn(q1[i], iq1[i]);
                auto row = [&](const float *m4, const float *v4, int n) {
                    const float4 x = *reinterpret_cast<const float4 *>(m4), y = *reinterpret_cast<const float4 *>(v4);
                    z = __fmaf_rn(-x.x, y.x, z);
                    if (n > 1) z = __fmaf_rn(-x.y, y.y, z);
                    if (n > 2) z = __fmaf_rn(-x.z, y.z, z);
                    if (n > 3) z = __fmaf_rn(-x.w, y.w, z);
                };
                if constexpr (DENSE) {  // the first block row has A Q^-1 = 0, B R^-1 = 0
#pragma unroll
                    for (int m = 0; m < NX; ++m)
                        z = __fadd_rn(z, __fmaf_rn(Qb[i * LD + m], q1[m], -__fmul_rn(Y[i * LD + m], qs[m])));
#pragma unroll
                    for (int m = 0; m < NU; m += 4) row(Bs + i * LB + m, rs + m, NU - m);
                    a.gamma[(size_t)kc * NX + i] = __fsub_rn(cv, z);
                } else {
#pragma unroll
                    for (int m = 0; m < NX; m += 4) row(X + i * LD + m, qs + m, NX - m);
#pragma unroll
                    for (int m = 0; m < NU; m += 4) row(Bm + i * LB + m, rs + m, NU - m);
                    a.gamma[(size_t)kc * NX + i] = first ? __fmaf_rn(-q1[i], iq1[i], cv) : __fsub_rn(cv, z);
                }
            }
        }
        __syncwarp();  // B and B R^-1 make room for D
        // the upper triangle as computed, the lower one mirrored
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
                const int i = ti + GR * r, jj = tj + GC * c;
                if (!DENSE && i == jj && i < NX) acc[r][c] += iq1[i];
            }
        if constexpr (F::SQUARE) {  // the mirrored entry sits in lane (tj, ti) as acc[c][r]
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int c = r; c < TC; ++c) {
                    const float up = __shfl_sync(0xffffffffu, acc[r][c], mirror);
                    if (c > r) acc[c][r] = up;
                    else if (ti > tj) acc[r][r] = up;
                }
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int c = 0; c < TC; ++c) M[r][c] = acc[r][c];
            put_strided(D, M);
        } else {
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int c = 0; c < TC; ++c) {
                    const int i = ti + GR * r, jj = tj + GC * c;
                    if (tile && i <= jj) {
                        D[i * LD + jj] = acc[r][c];
                        D[jj * LD + i] = acc[r][c];
                    }
                }
        }
    }
    __syncwarp();  // D complete; X (A) is free from here on
    if (mine) {
        block_out<NX, NX, LD, F::VW, GL>(a.Sd + (size_t)kc * NX * NX, D, t);
        if (!first) block_out<NX, NX, LD, F::VW, GL>(a.So + (size_t)j * NX * NX, Y, t, -1.f);
        if constexpr (NX == 36) {
            if (Sdp) pack_out(Sdp, D);
        }
    }

    // ---- Pd = D^-1: Gauss-Jordan without pivoting, symmetrised --------------------
    // The tile stays in registers (rows ti + GR r, columns tj + GC c); step p
    // passes row p and column p through shared memory (two parities, one warp
    // barrier).  p = GC c + x: the tile's row and column of the pivot are
    // fixed by c alone, so only c is unrolled.
    if constexpr (!F::SQUARE) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) M[r][c] = D[(tr + GR * r) * LD + tcb + GC * c];
    }
    gj_tile<F, NX>(M, rowb, colb, tr, tcb);
    {
        // X = (M + M^T) / 2
        if constexpr (F::SQUARE) {
            sym_tile<F>(M, mirror);
        } else {
            put_strided(X, M);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int c = 0; c < TC; ++c) M[r][c] = 0.5f * (M[r][c] + X[(tcb + GC * c) * LD + tr + GR * r]);
            __syncwarp();
        }
        put_strided(X, M);
    }
    __syncthreads();
    if (mine) {
        block_out<NX, NX, LD, F::VW, GL>(Pd + (size_t)kc * NX * NX, X, t);
        if constexpr (NX == 36) {
            if (Pdp) pack_out(Pdp, X);
        }
    }
    if (a.info && mine && bad) atomicOr(&a.info[b], MPCG_INFO_BADINPUT);

    // ---- Po = -Pd[k+1] (-(A Q^-1)[k+1] Pd[k]); the next group holds knot k + 1 ------
    const float *Xn = X, *Yn = Y;
    const bool has_next = mine && k + 1 < Nb;
    if (has_next) {
        Xn = X + WORDS;
        Yn = Y + WORDS;
    }
    nn(Yn, X, -1.f);
    put(D, 1.f);  // D is written out; its row stride covers the tile columns past nx
    __syncwarp();
    nn(Xn, D, 1.f);
    __syncwarp();
    put(D, -1.f);
    __syncwarp();
    if (has_next) block_out<NX, NX, LD, F::VW, GL>(Po + (size_t)(kc - b) * NX * NX, D, t);
}

// Recovery with dense costs, dz = G^-1 (C^T v - h), a half warp per knot: both
// blocks inverted by the tiled elimination, sums as in recover_dense_kernel
// (exact products, extended sums, one rounding).
template <int NX, int NU>
__global__ void __launch_bounds__(128)
recover_dense_tile_kernel(BatchView bv, const float *__restrict__ A, const float *__restrict__ B,
                          const float *__restrict__ Qf, const float *__restrict__ Rf, const float *__restrict__ hx,
                          const float *__restrict__ hu, const float *__restrict__ v, float *__restrict__ zx,
                          float *__restrict__ zu) {
    using F = FT<NX, NU>;
    static_assert(F::SQUARE && F::GL == 16, "half a warp per knot");
    constexpr int TR = F::TR, TC = F::TC, GR = F::GR, GC = F::GC, GL = F::GL, LD = F::LD, NP = F::NP, G = 128 / GL;
    __shared__ __align__(16) float sm[G][F::MAT + NU * LD + 2 * (F::ROWB + F::COLB) + 3 * NP];
    const int grp = threadIdx.x / GL, t = threadIdx.x % GL, ti = t / GC, tj = t % GC;
    float *Qi = sm[grp], *Ri = Qi + F::MAT, *rowb = Ri + NU * LD, *colb = rowb + 2 * F::ROWB, *vn = colb + 2 * F::COLB,
          *sx = vn + NP, *su = sx + NP;
    const int total = bv.total();
    if ((int)blockIdx.x * G >= total) return;
    const int kg = blockIdx.x * G + grp, kc = min(kg, total - 1);  // groups past the end store nothing
    const int b = bv.owner(kc);
    int k0, Nb;
    bv.range(b, k0, Nb);
    const bool last = kc - k0 + 1 >= Nb;
    const int j = kc - b, mirror = (threadIdx.x & 16) + tj * GC + ti;
    float M[TR][TC];
    auto load_tile = [&](const float *g, int n, bool on) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
                const int i = ti + GR * r, jj = tj + GC * c;
                M[r][c] = on && i < n && jj < n ? g[i * n + jj] : (i == jj ? 1.f : 0.f);
            }
    };
    auto put = [&](float *S, int n) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c)
                if (ti + GR * r < n && tj + GC * c < n) S[(ti + GR * r) * LD + tj + GC * c] = M[r][c];
    };
    if (t < NX) vn[t] = last ? 0.f : v[(size_t)(kc + 1) * NX + t];
    load_tile(Qf + (size_t)kc * NX * NX, NX, true);
    gj_tile<F, NX>(M, rowb, colb, ti, tj);
    sym_tile<F>(M, mirror);
    put(Qi, NX);
    load_tile(Rf + (last ? 0 : (size_t)j * NU * NU), NU, !last);
    gj_tile<F, NU>(M, rowb, colb, ti, tj);
    sym_tile<F>(M, mirror);
    put(Ri, NU);
    using AT = Acc<float>;
#pragma unroll
    for (int i0 = 0; i0 < NX + NU; i0 += GL) {
        const int i = i0 + t;
        const bool isx = i < NX;
        if (i >= NX + NU || (last && !isx)) continue;
        dfloat s = isx ? AT::add(AT::from(v[(size_t)kc * NX + i]), AT::from(-hx[(size_t)kc * NX + i]))
                       : AT::from(-hu[(size_t)j * NU + i - NX]);
        if (!last) {
            const float *col = isx ? A + (size_t)j * NX * NX + i : B + (size_t)j * NX * NU + i - NX;
            const int stride = isx ? NX : NU;
#pragma unroll
            for (int m = 0; m < NX; ++m) s = AT::add(s, AT::prod(-__ldg(col + m * stride), vn[m]));
        }
        (isx ? sx + i : su + i - NX)[0] = AT::to_T(s);
    }
    __syncwarp();
#pragma unroll
    for (int i0 = 0; i0 < NX + NU; i0 += GL) {
        const int i = i0 + t;
        const bool isx = i < NX;
        if (i >= NX + NU || kg >= total || (last && !isx)) continue;
        dfloat s = AT::zero();
        const float *row = isx ? Qi + i * LD : Ri + (i - NX) * LD, *x = isx ? sx : su;
        const int n = isx ? NX : NU;
        for (int m = 0; m < n; ++m) s = AT::add(s, AT::prod(row[m], x[m]));
        (isx ? zx + (size_t)kg * NX + i : zu + (size_t)j * NU + i - NX)[0] = AT::to_T(s);
    }
}

cudaError_t launch_recover_dense_14(BatchView bv, int Kgrid, const float *A, const float *B, const float *Qf,
                                    const float *Rf, const float *hx, const float *hu, const float *v, float *zx,
                                    float *zu, cudaStream_t s) {
    recover_dense_tile_kernel<14, 7><<<ceil_div(Kgrid, 8), 128, 0, s>>>(bv, A, B, Qf, Rf, hx, hu, v, zx, zu);
    return cudaGetLastError();
}

namespace {

template <int NX, int NU, bool DENSE>
cudaError_t launch_t(const SchurArgs<float> &a, float *Pd, float *Po, float *Sdp, float *Pdp, int sms, cudaStream_t s) {
    using F = FT<NX, NU>;
    // Few knots: spread them over the SMs (the chain of one knot is the time);
    // many: KPB_MAX per CTA, which repeats 1/KPB_MAX of the formations.
    const int kpb = std::min(F::KPB_MAX, std::max(1, ceil_div(a.Kgrid, sms > 0 ? sms : 1)));
    const int groups = ceil_div(kpb + 1, 32 / F::GL) * (32 / F::GL);
    const size_t smem = sizeof(float) * (size_t)(F::WORDS + (DENSE ? F::QWORDS : 0)) * groups;
    form_tile_kernel<NX, NU, DENSE><<<ceil_div(a.Kgrid, kpb), groups * F::GL, smem, s>>>(a, Pd, Po, Sdp, Pdp, kpb);
    return cudaGetLastError();
}

}  // namespace

// The two shapes above (dense costs: nx = 14), every block array aligned to
// its accesses (8 bytes at nx = 14, 16 at nx = 36).
bool form_tile_fits(const SchurArgs<float> &a, const float *Pd, const float *Po) {
    const bool s14 = a.nx == 14 && a.nu == 7, s36 = a.nx == 36 && a.nu == 12;
    if (!s14 && (!s36 || a.Qf)) return false;
    const uintptr_t bits = (uintptr_t)a.A | (uintptr_t)a.Sd | (uintptr_t)a.So | (uintptr_t)Pd | (uintptr_t)Po;
    return bits % (s14 ? 8 : 16) == 0;
}

cudaError_t launch_form_tile(const SchurArgs<float> &a, float *Pd, float *Po, float *Sdp, float *Pdp, int sms,
                             cudaStream_t s) {
    if (a.nx == 36) return launch_t<36, 12, false>(a, Pd, Po, Sdp, Pdp, sms, s);
    return a.Qf ? launch_t<14, 7, true>(a, Pd, Po, nullptr, nullptr, sms, s)
                : launch_t<14, 7, false>(a, Pd, Po, nullptr, nullptr, sms, s);
}

cudaError_t form_tile_prepare(int smem_optin) {
    auto one = [&](auto *fn) {
        cudaFuncAttributes fa;
        const cudaError_t e = cudaFuncGetAttributes(&fa, fn);
        if (e != cudaSuccess) return e;
        return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - (int)fa.sharedSizeBytes);
    };
    cudaError_t e = one(form_tile_kernel<14, 7, false>);
    if (e == cudaSuccess) e = one(form_tile_kernel<14, 7, true>);
    return e != cudaSuccess ? e : one(form_tile_kernel<36, 12, false>);
}

}  // namespace mpcg
