// Cluster PCG with one reduction per iteration (the recurrence, the exchanges
// and the parities are those of pcg_reg.cu) for float32 nx = 36 and float64
// nx = 14: a lane (or Q lanes) per row, and one warp of each CTA that only forms the sums.
//
// What bounds it.  float32, nx = 36: the exchanges and barriers, and the
// shared-memory reads (108 words of vector a row and product, 108 of Phi^-1).
// float64: each of an SM's four schedulers issues one FP64 instruction per 64
// cycles whatever its active lanes (measured; latency 66, a division 630), so
// the count of such instructions is the time: 42 per product and warp, and
// few warps, few additions and no repeated scalars beside them.  Therefore
//  - S p_old, which only the update needs, is formed by the row warps while the
//    sums of r~ travel, so it costs no time of its own;
//  - the sums of the accumulators are reduced by recursive halving (8 additions a
//    warp for five in place of 25);
//  - the last warp holds no rows: it adds the warp sums, exchanges them, forms
//    alpha and beta for everybody, and 1 / eta for the next beta while the
//    others update.
// Measured per iteration, against the general cluster kernel (pcg.cu, blocks in
// shared memory, two reductions): float32 nx = 36, N = 64: 1.89 against 8.4 us
// (N = 128: 2.99); float64 nx = 14, N = 101: 6.05 against 8.2 us, of which the
// three products' FP64 instructions are 3.9.
// Rows split over two or four lanes: slower at nx = 36 (N = 64, refined solve:
// 3.3 and 4.4 ms against 2.8: more warps read the vectors); in float64 faster
// while that fills schedulers without rows (N = 20: 4.0 against 6.1 us).
//
// Layout: CTA r of an instance's C <= 16 CTAs owns KPC = ceil(N/C) knots, thread
// (kl NX + i) Q + q part q of row i of its knot kl.  The row's 3 nx columns (blocks k-1, k, k+1)
// are consecutive words of a vector stored knot after knot.  The rows of S+ lie
// in registers; those of Phi^-1 too (float64) or in shared memory (float32, as
// 16-byte words, word w of all threads side by side).
#include <type_traits>

#include "pcg_sums.cuh"

namespace mpcg {

namespace {

constexpr int SPLIT_CMAX = 16;
constexpr int SPLIT_WMAX = 16;  // row warps that the warp sums have room for

struct SplitLayout {
    size_t vecR, vecP, vecZ, vec_bytes, halo, slot, wpart, scal, mbar, mail, misc, mats, total;
    // row_bytes > 0: the rows of Phi^-1 of `threads` threads too
    __host__ __device__ SplitLayout(int kpc_max, int nx, int esz, int threads, int row_bytes) {
        size_t o = 0;
        auto take = [&o](size_t bytes) {
            const size_t at = o;
            o += (bytes + 15) & ~size_t(15);
            return at;
        };
        vec_bytes = ((size_t)(kpc_max + 2) * nx * esz + 15) & ~size_t(15);
        vecR = take(vec_bytes);
        vecP = take(vec_bytes);
        vecZ = take(2 * vec_bytes);                  // by parity of the r~ exchange
        halo = take((size_t)2 * 2 * 2 * nx * esz);   // (S r~, S p) x parity x side
        slot = take(16 * 2 * 2 * SPLIT_CMAX + 8 * 2 * SPLIT_CMAX);  // parity x pair of sums x source CTA; the fifth: parity x source
        wpart = take(8 * 5 * SPLIT_WMAX);            // pair x warp; the fifth
        scal = take(48);
        mbar = take(sizeof(uint64_t) * 6);           // R0, R1, Z, T, peers stopped, instance mail
        mail = take(sizeof(int));
        misc = take(16);
        mats = take((size_t)row_bytes * threads);
        total = o;
    }
};

__device__ __forceinline__ void vec_load(const float *p, float (&o)[4]) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void vec_load(const double *p, double (&o)[2]) {
    const double2 v = *reinterpret_cast<const double2 *>(p);
    o[0] = v.x; o[1] = v.y;
}
__device__ __forceinline__ double sq_sum(double a, double, double) { return __dmul_rn(a, a); }
__device__ __forceinline__ float quot(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double quot(double a, double b) { return a / b; }

}  // namespace

// Q: lanes per row (float64), each with every Q-th pair of the columns
template <typename T, int NX, int MAXT, int Q = 1>
__global__ void __launch_bounds__(MAXT, 1) pcg_split_kernel(const PcgParams<T> P) {
    using AT = Acc<T>;
    using A = typename AT::type;
    constexpr bool PS = sizeof(T) == 4;                   // Phi^-1 in shared memory
    constexpr int ROW = 3 * NX, VW = 16 / (int)sizeof(T);  // a row, entries per 16-byte load
    constexpr int NCH = PS ? VW : 1;                       // chains of a product
    constexpr int WORDS = ROW / VW, WQ = (WORDS + Q - 1) / Q;  // 16-byte words of a row, of a lane
    static_assert(NX % VW == 0, "16-byte vector slots");
    static_assert(!PS || Q == 1, "whole rows");
    constexpr uint32_t R0 = 0, Z = 16, TT = 24, STOP = 32, MAIL = 40;  // mbarriers
    extern __shared__ __align__(16) unsigned char smem[];
    // float64: p_old^T S p_old as a fifth sum (2 % of the time, an FP64 addition more per
    // level); float32: carried, with the predicted beta g in eps (the fifth would take 7 %)
    constexpr bool FIFTH = sizeof(T) == 8;
    struct Sums {
        A eta, del, eps, old;  // r^T r~, r~^T S r~, (r~ + g / 2 p_old)^T S p_old, (FIFTH) p_old^T S p_old
        T rr;                  // ||r||^2
    };
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int nthreads = blockDim.x, W = nthreads / 32 - 1;  // row warps
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const bool sums = warp == W;  // the warp without rows
    const int kl = tid / (NX * Q), i = tid / Q % NX, q = tid % Q;

    const SplitLayout L(P.kpc_max, NX, sizeof(T), nthreads, PS ? ROW * (int)sizeof(T) : 0);
    T *vecR = reinterpret_cast<T *>(smem + L.vecR), *vecP = reinterpret_cast<T *>(smem + L.vecP);
    T *halo = reinterpret_cast<T *>(smem + L.halo), *scal = reinterpret_cast<T *>(smem + L.scal);
    A *wpart = reinterpret_cast<A *>(smem + L.wpart);
    int *mail = reinterpret_cast<int *>(smem + L.mail);
    int *flags = reinterpret_cast<int *>(scal + 4);
    int *s_abort = reinterpret_cast<int *>(smem + L.misc);  // set by a peer that gave up waiting
    volatile int *s_fail = s_abort + 1;                     // a warp of this CTA gave up waiting
    const uint32_t mb = smem_u32(smem + L.mbar);
    auto vecZ = [&](uint32_t par) { return reinterpret_cast<T *>(smem + L.vecZ + par * L.vec_bytes); };
    // halo rows of vector v (0: S r~, 1: S p), exchange parity, side (0: from
    // the left neighbour, 1: from the right)
    auto halo_off = [](int v, uint32_t par, int side) { return ((v * 2 + (int)par) * 2 + side) * NX; };

    if (tid == 0) {
        for (int m = 0; m < 6; ++m) mbar_init(mb + 8 * m, 8 * m == (int)STOP ? (C > 1 ? C - 1 : 1) : 1);
        *s_abort = 0;
        *s_fail = 0;
        for (int m = 0; m < 5 * SPLIT_WMAX; ++m) wpart[m] = AT::zero();
        fence_mbar_init();
    }
    cluster_sync_all();  // peers may push only after every mbarrier is initialised

    uint32_t xr = 0, xz = 0, mail_phase = 0;  // reductions, r~ exchanges (and S p exchanges) so far
    int served = 0;
    const bool has_left = rank > 0, has_right = rank + 1 < C;
    const uint32_t halo_bytes = (uint32_t)(NX * sizeof(T)) * ((has_left ? 1u : 0u) + (has_right ? 1u : 0u));

    for (;;) {
        // ---- the cluster's next instance (its first CTA draws) -------------------
        if (rank == 0 && tid == 0) {
            int b = -1;
            for (;;) {
                const int t = P.queue ? atomicAdd(P.queue, 1) : (int)(cluster_id_x() + (uint32_t)served++ * num_clusters_x());
                if (t >= P.n_tickets) {
                    b = -1;
                    break;
                }
                b = P.inst_list ? P.inst_list[t] : t;
                if (b < 0) break;  // ends the list for this cluster
                int k0, Nb;
                P.bv.range(b, k0, Nb);
                // an instance that is empty, flagged, or longer than the
                // launch was sized for is refused
                if (Nb >= 1 && ceil_div(Nb, C) <= P.kpc_max && !(P.info && P.info[b] != 0u)) break;
                if (P.stats && b < P.bv.B) {
                    mpcg_stats st{0, MPCG_BADINPUT, 0.0, 0.0};
                    P.stats[b] = st;
                }
            }
            for (int c = 0; c < C; ++c) st_async(map_rank(smem_u32(mail), c), __int_as_float(b), map_rank(mb + MAIL, c));
        }
        if (tid == 0) {
            mbar_arrive_expect(mb + MAIL, 4);
            if (!mbar_wait_bounded_abort(mb + MAIL, mail_phase, WAIT_LIMIT_NS, s_abort)) *s_fail = 1;
        }
        mail_phase ^= 1u;
        // Leaving after a wait gave up (here or in a peer), as in pcg_reg.cu
        auto leave = [&]() {
            if (tid == 0) cluster_drain(rank, C, smem_u32(s_abort), mb + STOP, DRAIN_LIMIT_NS, DRAIN_GRACE_NS);
            __syncthreads();
        };
        __syncthreads();
        if (*s_fail) {
            leave();
            return;
        }
        const int b = *mail;
        if (b < 0) break;

        int k0, Nb;
        P.bv.range(b, k0, Nb);
        const int c0 = k0 - b;
        const int KPC = ceil_div(Nb, C), kfirst = rank * KPC, k = kfirst + kl;
        const bool own = !sums && kl < KPC, active = own && k < Nb;  // row slot, row within the horizon
        const int max_iter = P.max_iter > 0 ? P.max_iter : 10 * Nb * NX;
        const int at = (kl + 1) * NX + i;  // this thread's row in a shared vector
        // the warps with a row of the first or last knot wait for the neighbours' rows
        const bool warp_edge = !sums && ((has_left && warp * 32 < NX * Q) ||
                                         (has_right && warp * 32 + 31 >= (KPC - 1) * NX * Q && warp * 32 < KPC * NX * Q));
        const bool one = own && q == 0;  // this row's only lane that writes or adds it
        const bool hleft = one && kl == 0 && has_left, hright = one && kl == KPC - 1 && has_right;
        const bool hany = hleft || hright, hboth = hleft && hright;
        const int side = hleft ? 0 : 1, hat = (side ? (KPC + 1) * NX : 0) + i;
        const uint32_t nb = map_rank(smem_u32(smem), hleft ? rank - 1 : (hright ? rank + 1 : rank));

        // ---- row i of S+ and Phi^-1 --------------------------------------------------
        // Phi^-1 rows without off-diagonal blocks: block Jacobi (precon 1), the
        // even knots' rows of the stair (2)
        const bool jac = P.precon == 1 || (P.precon == 2 && (k & 1) == 0);
        auto entry = [&](const T *Md, const T *Mo, bool off, int c) -> T {
            constexpr int n2 = NX * NX;
            const int blk = c / NX, j = c % NX;
            if (!active) return T(0);
            if (blk == 1) return __ldg(Md + (size_t)(k0 + k) * n2 + j * NX + i);
            if (!off) return T(0);
            if (blk == 0) return k >= 1 ? __ldg(Mo + (size_t)(c0 + k - 1) * n2 + i * NX + j) : T(0);
            return k + 1 < Nb ? __ldg(Mo + (size_t)(c0 + k) * n2 + j * NX + i) : T(0);
        };
        T sreg[WQ * VW], preg[PS ? 1 : WQ * VW];
        // entry e of this lane's part of the row is column col(e)
        auto col = [&](int e) { return ((e / VW) * Q + q) * VW + e % VW; };
        auto part = [&](const T *Md, const T *Mo, bool off, int e) -> T {
            return col(e) < ROW ? entry(Md, Mo, off, col(e)) : T(0);
        };
        float4 *mats = reinterpret_cast<float4 *>(smem + L.mats) + tid;
#pragma unroll
        for (int e = 0; e < WQ * VW; ++e) sreg[e] = part(P.Sd, P.So, true, e);
        if constexpr (PS) {
#pragma unroll
            for (int e = 0; e < ROW; e += 4)
                mats[(e / 4) * nthreads] = make_float4(entry(P.Pd, P.Po, !jac, e), entry(P.Pd, P.Po, !jac, e + 1),
                                                       entry(P.Pd, P.Po, !jac, e + 2), entry(P.Pd, P.Po, !jac, e + 3));
        } else {
#pragma unroll
            for (int e = 0; e < WQ * VW; ++e) preg[e] = part(P.Pd, P.Po, !jac, e);
        }

        // row . vec; float32 sums four chains, float64 one (its latency is
        // hardly above its issue interval)
        auto rowdot = [&](bool precon, const T *vec) -> T {
            T acc[NCH];
#pragma unroll
            for (int m = 0; m < NCH; ++m) acc[m] = T(0);
            const T *v = vec + kl * NX;
            if (active) {
#pragma unroll
                for (int j = 0; j < WQ; ++j) {
                    T x[VW], w[VW];
                    if ((j + 1) * Q > WORDS && j * Q + q >= WORDS) continue;  // past the row
                    vec_load(v + (j * Q + q) * VW, x);
                    if (PS && precon) vec_load(reinterpret_cast<const T *>(mats + j * nthreads), w);
#pragma unroll
                    for (int m = 0; m < VW; ++m)
                        acc[m % NCH] = fma_rn(precon ? (PS ? w[m] : preg[PS ? 0 : j * VW + m]) : sreg[j * VW + m], x[m], acc[m % NCH]);
                }
            }
            if constexpr (PS) return (acc[0] + acc[1]) + (acc[2] + acc[3]);
            T y = acc[0];
#pragma unroll
            for (int m = 1; m < Q; m *= 2) y += __shfl_xor_sync(0xffffffffu, y, m);
            return y;
        };
        // Boundary rows to offset off_l (off_r) of the left (right) neighbour's
        // shared memory; float32 rows leave in fours.
        auto push = [&](T y, uint32_t off_l, uint32_t off_r, uint32_t bar) {
            if (!warp_edge) return;
            const uint32_t mo = (uint32_t)L.mbar + bar, io = (uint32_t)sizeof(T) * (uint32_t)i;
            if constexpr (PS) {
                const float y1 = __shfl_down_sync(0xffffffffu, y, 1), y2 = __shfl_down_sync(0xffffffffu, y, 2),
                            y3 = __shfl_down_sync(0xffffffffu, y, 3);
                if (hany && i % 4 == 0) {
                    st_async_v4(nb + (hleft ? off_l : off_r) + io, y, y1, y2, y3, nb + mo);
                    if (hboth) {
                        const uint32_t nr = map_rank(smem_u32(smem), rank + 1);
                        st_async_v4(nr + off_r + io, y, y1, y2, y3, nr + mo);
                    }
                }
            } else {
                if (hany) st_async(nb + (hleft ? off_l : off_r) + io, y, nb + mo);
                if (hboth) {
                    const uint32_t nr = map_rank(smem_u32(smem), rank + 1);
                    st_async(nr + off_r + io, y, nr + mo);
                }
            }
        };
        // a row that leaves to the left is the receiver's halo from its right
        auto push_halo = [&](int v, uint32_t par, T y, uint32_t bar) {
            push(y, (uint32_t)(L.halo + sizeof(T) * halo_off(v, par, 1)), (uint32_t)(L.halo + sizeof(T) * halo_off(v, par, 0)), bar);
        };

        // ---- sums over the cluster of four (FIFTH: five) accumulators per row thread -----
        // A row warp reduces its own by recursive halving (lanes 8u hold sum u, lane 4
        // the fifth), leaves them and goes on.
        auto contribute = [&](A v0, A v1, A v2, A v3, A v4) {
            A x;
            if constexpr (FIFTH) {
                x = warp_sums5<AT>(v0, v1, v2, v3, v4);
                if (lane == 4) wpart[4 * SPLIT_WMAX + warp] = x;
            } else {
                x = halve<AT>(halve<AT>(v0, v2, 16), halve<AT>(v1, v3, 16), 8);
#pragma unroll
                for (int m = 4; m >= 1; m >>= 1) x = AT::add_tree(x, AT::shfl_xor(x, m));
            }
            const int u = lane >> 3;
            if ((lane & 7) == 0) wpart[(u >> 1) * 2 * SPLIT_WMAX + 2 * warp + (u & 1)] = x;
            named_bar_arrive(1, nthreads);
        };
        // The sums warp adds the warps', pushes the CTA's to every CTA (lanes 0-15 the
        // first pair of sums, 16-31 the second, 0-15 the fifth) and adds those of all.
        auto collect = [&](uint32_t nh) -> Sums {
            const uint32_t par = xr & 1u, bar = mb + R0 + 8 * par;
            const int c16 = lane & 15, pr = lane >> 4, w8 = lane & 7;
            const uint32_t fifth_off = (uint32_t)L.slot + (uint32_t)(16 * 2 * 2 * SPLIT_CMAX + 8 * SPLIT_CMAX * (int)par);
            const uint32_t slot_off = (uint32_t)L.slot + (uint32_t)((((int)par * 2 + pr) * SPLIT_CMAX) * 16);
            if (C > 1 && lane == 0) mbar_arrive_expect(bar, (uint32_t)C * (FIFTH ? 40u : 32u) + nh * halo_bytes);
            const uint32_t pb = map_rank(smem_u32(smem), c16 < C ? c16 : 0);
            named_bar_sync(1, nthreads);
            A x, y0, y1, y2 = AT::zero();
            if constexpr (FIFTH) {  // sum lane / 8 of row warp lane % 8: three additions for all five
                static_assert(!FIFTH || MAXT <= 288, "at most 8 row warps");
                const int u = lane >> 3;
                x = fold5<AT>(wpart[(u >> 1) * 2 * SPLIT_WMAX + 2 * w8 + (u & 1)], wpart[4 * SPLIT_WMAX + w8]);
                y0 = bcast(x, 16 * pr);
                y1 = bcast(x, 16 * pr + 8);
                y2 = bcast(x, 4);
            } else {
                const A *w = wpart + pr * 2 * SPLIT_WMAX + 2 * w8;
                load_pair(w, y0, y1);
                if (W > 8) {
                    A z0, z1;
                    load_pair(w + 16, z0, z1);
                    y0 = AT::add_tree(y0, z0);
                    y1 = AT::add_tree(y1, z1);
                }
#pragma unroll
                for (int m = 4; m >= 1; m >>= 1) {
                    y0 = AT::add_tree(y0, AT::shfl_xor(y0, m));
                    y1 = AT::add_tree(y1, AT::shfl_xor(y1, m));
                }
                x = lane & 8 ? y1 : y0;
            }
            if (C > 1) {
                const uint32_t pbar = pb + (uint32_t)L.mbar + R0 + 8 * par;
                if (c16 < C) push_pair(pb + slot_off + 16u * (uint32_t)rank, y0, y1, pbar);
                if (FIFTH && lane < C) st_async(pb + fifth_off + 8u * (uint32_t)rank, y2, pbar);
                if (warp_wait(bar, (xr >> 1) & 1u, s_abort)) *s_fail = 1;
                y0 = y1 = y2 = AT::zero();
                if (c16 < C) {
                    load_pair(reinterpret_cast<const A *>(smem + slot_off + 16 * c16), y0, y1);
                    if (FIFTH) y2 = *reinterpret_cast<const A *>(smem + fifth_off + 8 * c16);
                }
                x = halve<AT>(y0, y1, 8);
                if constexpr (FIFTH) {
                    x = fold5<AT>(x, AT::add_tree(y2, AT::shfl_xor(y2, 8)));
                } else {
#pragma unroll
                    for (int m = 4; m >= 1; m >>= 1) x = AT::add_tree(x, AT::shfl_xor(x, m));
                }
            }
            Sums r;
            r.old = FIFTH ? bcast(x, 4) : AT::zero();
            const T xf = AT::to_T(x);
            r.eta = bcast(x, 0);
            r.rr = __shfl_sync(0xffffffffu, xf, 8);
            r.del = bcast(x, 16);
            r.eps = bcast(x, 24);
            return r;
        };

        // ---- initialisation: r = b - S lambda0, ||b||^2 -------------------------------
        for (int e = tid; e < (int)(4 * L.vec_bytes / sizeof(T)); e += nthreads) vecR[e] = T(0);  // R, P and both Z
        __syncthreads();
        T lam = T(0), r = T(0), p = T(0), s = T(0), bv = T(0);
        T *v0 = vecZ(0);
        if (active) {
            lam = P.lam[(size_t)(k0 + k) * NX + i];
            bv = P.rhs_sign * P.rhs[(size_t)(k0 + k) * NX + i];
            if (one) v0[at] = lam;
        }
        // lambda0 halo straight from global memory
        if (one && kl == 0 && kfirst >= 1 && kfirst - 1 < Nb) v0[i] = P.lam[(size_t)(k0 + kfirst - 1) * NX + i];
        if (one && kl == KPC - 1 && kfirst + KPC < Nb) v0[(KPC + 1) * NX + i] = P.lam[(size_t)(k0 + kfirst + KPC) * NX + i];
        __syncthreads();
        if (active) {
            A a = AT::from(bv);
            // (the blocks once more from memory: an index that is not fixed at
            // compile time would take sreg out of the registers)
#pragma unroll 4
            for (int e = 0; e < ROW; ++e) a = AT::add(a, AT::prod(-entry(P.Sd, P.So, true, e), v0[kl * NX + e]));
            r = AT::to_T(a);
        }
        if (one) vecR[at] = r;
        __syncthreads();
        for (int e = tid; e < (int)(L.vec_bytes / sizeof(T)); e += nthreads) v0[e] = T(0);
        const bool mode1 = P.tol_mode == 1;
        const uint32_t ipar = xr & 1u;
        A bb = AT::zero(), eta = AT::zero();
        T tol_t = T(0);
        if (sums) {
            const double tol = P.tol > 0 ? P.tol : 1e-6;
            bb = collect(1u).eta;
            tol_t = mode1 ? (T)tol : (T)(tol * tol * AT::to_double(bb));
        } else {
            push_halo(0, ipar, r, R0 + 8 * ipar);
            contribute(one ? AT::prod(bv, bv) : AT::zero(), AT::zero(), AT::zero(), AT::zero(), AT::zero());
        }
        ++xr;
        __syncthreads();
        bool timed_out = *s_fail != 0;
        if (hany) vecR[hat] = halo[halo_off(0, ipar, side) + i];
        if (hboth) vecR[2 * NX + i] = halo[halo_off(0, ipar, 1) + i];
        __syncthreads();

        const T big = sizeof(T) == 4 ? (T)3.402823466e38f : (T)1.7976931348623157e308;
        A acc = AT::zero();     // p^T S p; this, rr and recip the sums warp's
        T rr = T(0), g = T(0);  // g (every warp's): the last beta (FIFTH: 0)
        EtaRecip<T> recip;
        int iters = 0;
        bool broke = false, late = false;  // late: this warp gave up waiting for S p rows
        for (int it = 0; !timed_out; ++it) {
            const uint32_t zpar = xz & 1u, rpar = xr & 1u;  // halo rows alternate once per iteration
            if (late) *s_fail = 1;  // read after the second barrier from here
            T *vz = vecZ(zpar);
            T z = T(0), qv = T(0), t = T(0), hz = T(0), hp = T(0), hr = T(0);
            A s_eta = AT::zero(), s_rr = AT::zero(), s_eps = AT::zero(), s_old = AT::zero();
            // ---- r~ = Phi^-1 r, boundary rows to the neighbours -----------------------
            if (!sums) {
                z = rowdot(true, vecR);
                push(z, (uint32_t)(L.vecZ + zpar * L.vec_bytes + sizeof(T) * (KPC + 1) * NX), (uint32_t)(L.vecZ + zpar * L.vec_bytes), Z);
                if (one) vz[at] = z;
                if (Q == 1 || one) {
                    s_eta = AT::prod(r, z);
                    s_rr = sq_sum(r, T(0), A{});
                    s_eps = AT::prod(FIFTH ? z : fma_rn(T(0.5) * g, p, z), s);
                    if (FIFTH) s_old = AT::prod(p, s);
                }
            } else {
                if (C > 1 && lane == 0) {
                    mbar_arrive_expect(mb + Z, halo_bytes);
                    mbar_arrive_expect(mb + TT, halo_bytes);
                }
                if (it > 0) recip.set(AT::to_T(eta));
            }
            __syncthreads();
            if (!sums) {
                // ---- S r~, its sums, then S p_old while they travel ---------------------
                if (warp_edge)
                    if (warp_wait(mb + Z, xz & 1u, s_abort)) *s_fail = 1;
                qv = rowdot(false, vz);
                push_halo(0, zpar, qv, R0 + 8 * rpar);
                contribute(s_eta, s_rr, Q == 1 || one ? AT::prod(z, qv) : AT::zero(), s_eps, s_old);
                t = rowdot(false, vecP);
                push_halo(1, zpar, t, TT);
                if (hany) {
                    hz = vz[hat];
                    hp = vecP[hat];
                    hr = vecR[hat];
                }
            } else {
                // ---- alpha, beta and the exit tests, in T from the extended sums ---------
                const Sums S = collect(1u);
                const T etan = AT::to_T(S.eta);
                const T beta = recip.beta(etan, AT::to_T(eta));  // 0 in the first iteration
                if (FIFTH) acc = S.old;
                const A old = acc;
                acc = curvature(S.del, S.eps, acc, beta, g);
                const T ups = rounded(acc, T(0)), alpha = quot(etan, ups);
                eta = S.eta;
                rr = S.rr;
                const bool done = !(fabs(etan) <= big && rr <= big) || (mode1 ? etan < tol_t : rr <= tol_t) || it >= max_iter;
                const bool direct = doubtful(ups, S.del, S.eps, old, beta, g);
                if (lane == 0) {
                    scal[0] = alpha;
                    scal[1] = beta;
                    *flags = (done ? 1 : 0) | (direct ? 2 : 0);
                }
            }
            ++xr;
            iters = it;
            __syncthreads();
            if (*s_fail) {  // every warp saw the same
                timed_out = true;
                break;
            }
            const T beta = scal[1];
            T alpha = scal[0];
            const int f = *flags;
            if (f & 1) break;
            if (!FIFTH) g = beta;
            // p = r~ + beta p, S p = S r~ + beta S p_old, lambda += alpha p,
            // r -= alpha S p; the halo copies of p and r alike
            s = fma_rn(beta, t, qv);
            p = fma_rn(beta, p, z);
            if (f & 2) {  // sum p^T S p itself
                __syncthreads();  // flags and scalars are read
                if (sums) {
                    acc = collect(0u).eta;
                    const T ud = AT::to_T(acc);
                    if (lane == 0) {
                        scal[0] = AT::div(AT::to_T(eta), ud);
                        *flags = !(ud > T(0)) || !(ud <= big);
                    }
                } else {
                    contribute(Q == 1 || one ? AT::prod(p, s) : AT::zero(), AT::zero(), AT::zero(), AT::zero(), AT::zero());
                }
                ++xr;
                __syncthreads();
                if (*s_fail) {
                    timed_out = true;
                    break;
                }
                if (*flags) {
                    broke = true;
                    iters = it + 1;
                    break;
                }
                alpha = scal[0];
            }
            if (!sums) {
                r = fma_rn(-alpha, s, r);
                lam = fma_rn(alpha, p, lam);
                if (one) {
                    vecR[at] = r;
                    vecP[at] = p;
                }
                if (warp_edge)
                    late = warp_wait(mb + TT, xz & 1u, s_abort);
                if (hany) {
                    const T sh = fma_rn(beta, halo[halo_off(1, zpar, side) + i], halo[halo_off(0, zpar, side) + i]);
                    vecR[hat] = fma_rn(-alpha, sh, hr);
                    vecP[hat] = fma_rn(beta, hp, hz);
                }
                if (hboth) {
                    T *vr = vecR + 2 * NX + i, *vp = vecP + 2 * NX + i;
                    *vr = fma_rn(-alpha, fma_rn(beta, halo[halo_off(1, zpar, 1) + i], halo[halo_off(0, zpar, 1) + i]), *vr);
                    *vp = fma_rn(beta, *vp, vz[2 * NX + i]);
                }
            }
            ++xz;
            __syncthreads();
        }
        // the S p rows of the last iteration are still to be taken in
        if (!timed_out) {
            if (warp_edge && warp_wait(mb + TT, xz & 1u, s_abort)) *s_fail = 1;
            ++xz;
        }
        // ---- write back --------------------------------------------------------------
        if (active && one) P.lam[(size_t)(k0 + k) * NX + i] = lam;
        if (rank == 0 && sums && lane == 0 && P.stats) {
            const T etan = AT::to_T(eta);
            mpcg_stats st;
            st.iters = iters;
            st.status = timed_out ? MPCG_TIMEOUT
                        : broke   ? MPCG_BREAKDOWN
                        : !(isfinite(etan) && isfinite(rr))    ? MPCG_NONFINITE
                        : (mode1 ? etan < tol_t : rr <= tol_t) ? MPCG_CONVERGED
                                                               : MPCG_NOT_CONVERGED;
            st.eta = AT::to_double(eta);
            const double bbd = AT::to_double(bb), rrd = (double)rr;
            st.relres = bbd > 0.0 ? sqrt(rrd / bbd) : sqrt(rrd);
            P.stats[b] = st;
        }
        __syncthreads();
        if (*s_fail) {
            leave();
            return;
        }
    }
    cluster_sync_all();  // peers may push into this CTA's shared memory until they leave too
}

namespace {

// Variants by registers: two warps per scheduler leave 255 a thread, three 168.
// float32 nx = 36: up to 6 knots (8 warps with the sums warp), up to 8 (10);
// float64 nx = 14: up to 16 knots (8).
template <typename T>
struct SplitForm;
template <>
struct SplitForm<float> {
    static constexpr int NX = 36, KPC_MAX = 8, ROW_BYTES = 3 * 36 * 4;
    static int lanes(int) { return 1; }
    static int variant(int kpc) { return kpc <= 6 ? 1 : 2; }
    static auto fn(int v) { return v == 1 ? pcg_split_kernel<float, 36, 256> : pcg_split_kernel<float, 36, 320>; }
};
template <>
struct SplitForm<double> {
    static constexpr int NX = 14, KPC_MAX = 16, ROW_BYTES = 0;
    // Lanes per row, so that a product's instructions spread over the four
    // schedulers (8 knots x 2 lanes: 7 warps).  Per iteration with 1 lane -> as
    // chosen: N = 20 6.1 -> 4.0 us, 50 6.0 -> 4.6, 64 5.9 -> 4.5, 96 5.9 -> 5.4, 101
    // 6.0 -> 5.9 (4 lanes at 3-4 knots: 4.5-4.8, 1 at 5: no gain over 6.0); the fifth
    // sum, added since, takes 0.1-0.2.
    static int lanes(int kpc) { return kpc <= 2 ? 4 : kpc <= 8 ? 2 : 1; }
    static int variant(int kpc) { return lanes(kpc); }
    static auto fn(int v) {
        return v == 4 ? pcg_split_kernel<double, 14, 256, 4> : v == 2 ? pcg_split_kernel<double, 14, 256, 2> : pcg_split_kernel<double, 14, 256>;
    }
};

cudaLaunchConfig_t split_config(const PcgLaunch &L, int clusters, cudaLaunchAttribute *attr, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.C * clusters, 1, 1);
    cfg.blockDim = dim3(L.threads, 1, 1);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = L.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

template <typename T>
int pcg_split_shape(int nx, int N, int C, PcgLaunch &L) {
    using F = SplitForm<T>;
    const int kpc = ceil_div(N, C);
    if (nx != F::NX || kpc > F::KPC_MAX) return 0;
    L.cta_mode = 0;
    L.split_rows = F::variant(kpc);
    L.C = C;
    L.kpc_max = kpc;
    L.threads = 32 * (ceil_div(kpc * F::NX * F::lanes(kpc), 32) + 1);
    L.smem = SplitLayout(kpc, nx, sizeof(T), L.threads, F::ROW_BYTES).total;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = split_config(L, 1, attr, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, F::fn(L.split_rows), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <typename T>
cudaError_t pcg_split_launch(const PcgLaunch &L, const PcgParams<T> &P0, cudaStream_t s) {
    PcgParams<T> P = P0;
    P.kpc_max = L.kpc_max;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = split_config(L, L.clusters, attr, s);
    return cudaLaunchKernelEx(&cfg, SplitForm<T>::fn(L.split_rows), P);
}

cudaError_t pcg_split_prepare(int smem_optin) {
    auto one = [&](auto *fn) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
    };
    cudaError_t e = one(SplitForm<float>::fn(1));
    if (e == cudaSuccess) e = one(SplitForm<float>::fn(2));
    for (int v : {1, 2, 4})
        if (e == cudaSuccess) e = one(SplitForm<double>::fn(v));
    return e;
}

template int pcg_split_shape<float>(int, int, int, PcgLaunch &);
template int pcg_split_shape<double>(int, int, int, PcgLaunch &);
template cudaError_t pcg_split_launch<float>(const PcgLaunch &, const PcgParams<float> &, cudaStream_t);
template cudaError_t pcg_split_launch<double>(const PcgLaunch &, const PcgParams<double> &, cudaStream_t);

}  // namespace mpcg
