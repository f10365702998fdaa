// Register-resident, thread-block-cluster PCG for float32, nx = 14
// (Algorithm 1, organised per block row as in Algorithm 2 of the paper), with
// ONE cluster-wide reduction per iteration.
//
// What bounds it: the operators never leave the SMs, so an iteration costs
// what its exchanges and CTA barriers cost.  Algorithm 1 as printed has two
// dependent reductions (p^T S p for alpha; r^T r~ and ||r||^2 for beta and the
// exit).  Since p = r~ + beta p_old,
//     p^T S p = r~^T S r~ + 2 beta r~^T (S p_old) + beta^2 p_old^T S p_old,
// so alpha needs only sums that are known once r~ and S r~ are: one reduction
// of (r^T r~, ||r||^2, r~^T S r~, r~^T S p_old) serves both scalars.  The
// identity uses only the symmetry of S+ (not orthogonality of the residuals,
// nor symmetry of Phi^-1), and S p = S r~ + beta S p_old takes S p_old from a
// fresh product of the stored p each iteration, so no error is carried from
// one iteration to the next: emulated in float32 on the Kuka-shaped problems
// (N = 32..512, cold and warm), iteration counts equal Algorithm 1's and
// lambda differs from it by what another summation order changes (1e-6 warm).
// The Chronopoulos-Gear form, which carries S p by recurrence, is 3 to 10
// times further off.  The price is a third product, 84 FMAs per lane, which
// runs while the boundary rows of r~ travel to the neighbour CTAs.  Where the
// identity cancels (p^T S p below 1/16 of r~^T S r~; 0.29 was the smallest
// share seen on the emulated problems) the sum p^T S p is taken directly with
// one more reduction.  Measured on GB300 at fixed iteration counts: 1.75 us
// per iteration at N = 512 (16 CTAs x 32 knots) and 1.50 at N = 128 (16 x 8)
// against 2.23 and 1.98 with two reductions.  Of the 1.75 us, by leaving parts
// out one at a time: the three products 0.2-0.3 each (bound by the shared-
// memory reads of the vectors, 128 bytes per clock), the warp sums 0.11, the
// CTA sums 0.11, the sums over CTAs 0.06; the rest is the transport (0.12 one
// way) and the CTA barriers.
//
// Launch shape: clusters of C <= 16 CTAs; a group of G CTAs (the whole
// cluster, or a power-of-two part of it, below) solves one instance; CTA r of
// the group owns knots [r KPC, (r+1) KPC), KPC = ceil(N/G) <= 32; 8 lanes own
// a knot, lanes 0..6 two adjacent rows each, and keep their rows of S+ and
// Phi^-1 (2 x 84 floats) in registers for the whole solve.  r, p, r~ (with
// one halo knot on each side) live in shared memory.
//
// PS form: with many instances the exchanges of one leave the SM idle two
// thirds of the time, and one 16-CTA cluster per GPC leaves SMs unused, so two
// CTAs share an SM: 128 registers a thread hold the rows of S+, the rows of
// Phi^-1 lie in shared memory (same products in the same order).  The shared-
// memory reads then bound it: an iteration takes 1.84 times as long.
//
// Groups: a launch with more instances than clusters splits its clusters as
// the long instances run out.  At level l a group of C >> l CTAs takes only
// instances that need more than half of it at 32 knots per CTA; when that
// class is exhausted the group splits in two.  A ragged batch then runs its
// long horizons first, and short ones do not occupy a whole cluster (256
// instances of 32..512 knots: 42.8 ms with a 16-CTA cluster for each and two
// reductions, 27.5 ms split, 25.3 with two CTAs per SM).
//
// Stages: a GPC holds one or two clusters of 16 and then has SMs to spare (14
// clusters, 224 of 304 CTAs, with two CTAs per SM), and 257..384 knots need no
// 16.  So a batch of more than one wave takes up to three launches, for the
// horizons that need full clusters (16, 8 or 4 CTAs), those that 3/4 hold and those
// that half holds (which split); each may begin in the SMs that the one before
// leaves free.  One launch -> stages: 256 instances of 32..512 knots 25.5 -> 19.9
// ms, 64 of 150 3.69 -> 2.27, 40 of 260..384 6.37 -> 4.45, 64 of 65..96 0.95 -> 0.91;
// where all instances need the full size, nothing (256 of 120..128: 4.90 -> 5.03).
// 13 CTAs for the middle stage fit the GPU worse (20.9).
//
// Exchanges (st.async pushes completing transaction bytes on the receiver's
// mbarriers, no cluster barrier in the loop): per iteration the boundary rows
// of r~ go to the neighbour CTAs (barrier Z), then each CTA's four sums go to
// every CTA of the group together with the boundary rows of S r~ and S p_old
// (barrier R).  Buffers alternate by exchange parity: a peer can be at most
// one reduction ahead, since the next one needs this CTA's sums.  All CTAs
// add the partial sums in the same order, so they take identical decisions;
// halo copies of r and p are updated with the owner's own multiply-adds.
#include <climits>
#include <type_traits>

#include "pcg_sums.cuh"

namespace mpcg {

namespace {

constexpr int NXR = 14;   // block size
constexpr int VSR = 16;   // floats per knot slot of a shared vector
constexpr int LPR = 8;    // lanes per knot
constexpr int CMAX = 16;  // CTAs per cluster
constexpr int WMAX = 8;   // warps per CTA
constexpr int PROWS = 3 * 2 * NXR;  // a thread's entries of one operator
constexpr int LEVELS = 5; // group sizes C, C/2, ..., C/16

// Shared-memory carve-up, in bytes; the same on host and device.
struct RegLayout {
    size_t vecR, vecP, vecZ, halo, slot, wpart, mbar, mail, misc, mats, total;
    // threads > 0: the rows of Phi^-1 of so many threads too
    __host__ __device__ RegLayout(int kpc_max, int threads) {
        size_t o = 0;
        auto take = [&o](size_t bytes) {
            const size_t at = o;
            o += (bytes + 15) & ~size_t(15);
            return at;
        };
        const size_t vec = sizeof(float) * (size_t)(kpc_max + 2) * VSR;
        vecR = take(vec);
        vecP = take(vec);
        vecZ = take(vec);
        halo = take(sizeof(float) * 3 * 2 * 2 * VSR);  // (r~, S r~, S p) x parity x side
        slot = take(16 * 2 * 2 * CMAX);                // parity x pair of sums x source CTA
        wpart = take(8 * 4 * WMAX);                    // sum x warp
        mbar = take(sizeof(uint64_t) * (4 + LEVELS));  // R0, R1, Z, peers stopped, instance mail
        mail = take(sizeof(int) * LEVELS);
        misc = take(16);
        mats = take(sizeof(float) * (size_t)PROWS * threads);
        total = o;
    }
};

// Two rows of one block row times the halo'd vector: the knot's three
// 16-float vector slots are read once for both rows.
__device__ __forceinline__ void rowdot2(const float (&d)[2][NXR], const float (&l)[2][NXR],
                                        const float (&u)[2][NXR], const float *vprev,
                                        const float *vself, const float *vnext, float (&y)[2]) {
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, b0 = 0.f, b1 = 0.f, b2 = 0.f;
    const float4 *s4 = reinterpret_cast<const float4 *>(vself);
    const float4 *p4 = reinterpret_cast<const float4 *>(vprev);
    const float4 *n4 = reinterpret_cast<const float4 *>(vnext);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 xs = s4[q], xp = p4[q], xn = n4[q];
        const float vs_[4] = {xs.x, xs.y, xs.z, xs.w};
        const float vp_[4] = {xp.x, xp.y, xp.z, xp.w};
        const float vn_[4] = {xn.x, xn.y, xn.z, xn.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int j = 4 * q + t;
            if (j < NXR) {
                a0 = __fmaf_rn(d[0][j], vs_[t], a0);
                b0 = __fmaf_rn(d[1][j], vs_[t], b0);
                a1 = __fmaf_rn(l[0][j], vp_[t], a1);
                b1 = __fmaf_rn(l[1][j], vp_[t], b1);
                a2 = __fmaf_rn(u[0][j], vn_[t], a2);
                b2 = __fmaf_rn(u[1][j], vn_[t], b2);
            }
        }
    }
    y[0] = (a0 + a1) + a2;
    y[1] = (b0 + b1) + b2;
}

// The same with the thread's rows in shared memory (PS form): 21 four-entry
// words per thread, word c of all threads side by side, so a warp's load is
// conflict-free; per block seven words, the two rows' entries 4 q .. 4 q + 3
// in turn (the last word: entries 12 and 13 of both).
__device__ __forceinline__ void rowdot2_ps(const float4 *m, int stride, const float *vprev,
                                           const float *vself, const float *vnext, float (&y)[2]) {
    float sum[3][2];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const float4 *v4 = reinterpret_cast<const float4 *>(b == 0 ? vself : b == 1 ? vprev : vnext);
        const float4 *w = m + (size_t)7 * b * stride;
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 x = v4[q], r0 = w[2 * q * stride], r1 = w[(2 * q + 1) * stride];
            a0 = __fmaf_rn(r0.x, x.x, a0);
            a1 = __fmaf_rn(r1.x, x.x, a1);
            a0 = __fmaf_rn(r0.y, x.y, a0);
            a1 = __fmaf_rn(r1.y, x.y, a1);
            a0 = __fmaf_rn(r0.z, x.z, a0);
            a1 = __fmaf_rn(r1.z, x.z, a1);
            a0 = __fmaf_rn(r0.w, x.w, a0);
            a1 = __fmaf_rn(r1.w, x.w, a1);
        }
        const float2 x = *reinterpret_cast<const float2 *>(v4 + 3);
        const float4 r = w[6 * stride];
        a0 = __fmaf_rn(r.x, x.x, a0);
        a1 = __fmaf_rn(r.z, x.x, a1);
        sum[b][0] = __fmaf_rn(r.y, x.y, a0);
        sum[b][1] = __fmaf_rn(r.w, x.y, a1);
    }
    y[0] = (sum[0][0] + sum[1][0]) + sum[2][0];
    y[1] = (sum[0][1] + sum[1][1]) + sum[2][1];
}

__device__ __forceinline__ float resid_row(float b, const float (&d)[NXR], const float (&l)[NXR],
                                           const float (&u)[NXR], const float *vprev,
                                           const float *vself, const float *vnext) {
    dfloat a{b, 0.f};
#pragma unroll
    for (int j = 0; j < NXR; ++j) {
        a = df_add(a, df_prod(-d[j], vself[j]));
        a = df_add(a, df_prod(-l[j], vprev[j]));
        a = df_add(a, df_prod(-u[j], vnext[j]));
    }
    return __fadd_rn(a.hi, a.lo);
}

}  // namespace

template <typename AT, bool PS>
__global__ void __launch_bounds__(32 * WMAX, PS ? 2 : 1) pcg_reg_kernel(const PcgParams<float> P) {
    using A = typename AT::type;
    static_assert(sizeof(A) == 8, "sums travel in pairs of 8 bytes");
    extern __shared__ __align__(16) unsigned char smem[];
    struct Sums {
        A eta;               // r^T r~
        float rr, del, eps;  // ||r||^2, r~^T S r~, r~^T S p_old
    };

    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int nthreads = blockDim.x, W = nthreads / 32;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int kl = tid / LPR, li = tid % LPR;

    const RegLayout L(P.kpc_max, PS ? blockDim.x : 0);
    float *vecR = reinterpret_cast<float *>(smem + L.vecR);
    float *vecP = reinterpret_cast<float *>(smem + L.vecP);
    float *vecZ = reinterpret_cast<float *>(smem + L.vecZ);
    float *halo = reinterpret_cast<float *>(smem + L.halo);
    unsigned char *slots = smem + L.slot;
    A *wpart = reinterpret_cast<A *>(smem + L.wpart);
    int *mail = reinterpret_cast<int *>(smem + L.mail);
    int *s_abort = reinterpret_cast<int *>(smem + L.misc);  // set by a peer that gave up waiting
    volatile int *s_fail = s_abort + 1;                     // a warp of this CTA gave up waiting
    const uint32_t mb = smem_u32(smem + L.mbar);
    const uint32_t mbZ = mb + 16, mbS = mb + 24;
    // halo slot of vector v (0: r~, 1: S r~, 2: S p), exchange parity, side
    // (0: from the left neighbour, 1: from the right), in floats
    auto halo_off = [](int v, uint32_t par, int side) { return ((v * 2 + (int)par) * 2 + side) * VSR; };

    if (tid == 0) {
        for (int i = 0; i < 4 + LEVELS; ++i) mbar_init(mb + 8 * i, i == 3 ? (C > 1 ? C - 1 : 1) : 1);
        *s_abort = 0;
        *s_fail = 0;
        for (int i = 0; i < 4 * WMAX; ++i) wpart[i] = AT::zero();
        fence_mbar_init();
    }
    cluster_sync_all();  // peers may push only after every mbarrier is initialised

    const int arm = 32 * (W / 2);   // the thread that arms the barriers: not in a boundary warp
    int wpow = 1;                   // warps, rounded up to a power of two
    while (wpow < W) wpow <<= 1;
    uint32_t xr = 0, xz = 0;        // reductions and r~ exchanges done so far (parities, phases)
    int fail = 0;                   // this warp gave up a wait
    bool timed_out = false;
    int level = 0, g0 = 0, G = C;   // this CTA's group: ranks [g0, g0 + G)
    uint32_t mail_phase = 0;
    int served = 0;
    grid_dep_launch();
    // the next stage overlaps this one, so the last must outlive them all: one
    // thread of each stage leaves only when the stage before it is complete
    auto leave = [&]() {
        if (blockIdx.x == 0 && tid == 0) grid_dep_wait();
    };

    for (;;) {
        const int gr = rank - g0;  // rank in the group
        const bool has_left = gr > 0, has_right = gr + 1 < G;

        // ---- the group's next instance (its first CTA draws) -----------------
        if (gr == 0 && tid == 0) {
            int b = -1;
            for (;;) {
                const int t = P.queue ? atomicAdd(P.queue + level, 1)
                                      : (int)(cluster_id_x() + (uint32_t)served++ * num_clusters_x());
                if (t >= P.n_tickets) break;
                b = P.inst_list ? P.inst_list[t] : t;
                if (b < 0) {  // ends the list for this group
                    b = -2;
                    break;
                }
                int k0, Nb;
                P.bv.range(b, k0, Nb);
                if (Nb <= P.n_above || Nb > P.n_upto) {  // another stage's instance
                    b = -1;
                    continue;
                }
                const bool fits = Nb >= 1 && ceil_div(Nb, C) <= P.kpc_max;
                if (P.split) {  // another level's instance?
                    int need = C, l = 0;
                    while (fits && need > 1 && ceil_div(Nb, need / 2) <= P.kpc_max) {
                        need /= 2;
                        ++l;
                    }
                    if (l != level) {
                        b = -1;
                        continue;
                    }
                }
                // an instance that is empty, flagged, or longer than the
                // launch was sized for is refused
                if (fits && !(P.info && P.info[b] != 0u)) break;
                if (P.stats && b < P.bv.B) {
                    mpcg_stats st{0, MPCG_BADINPUT, 0.0, 0.0};
                    P.stats[b] = st;
                }
                b = -1;
            }
            for (int q = 0; q < G; ++q)
                st_async(map_rank(smem_u32(&mail[level]), g0 + q), __int_as_float(b), map_rank(mb + 8 * (4 + level), g0 + q));
        }
        if (tid == 0) {
            mbar_arrive_expect(mb + 8 * (4 + level), 4);
            fail = !mbar_wait_bounded_abort(mb + 8 * (4 + level), mail_phase, WAIT_LIMIT_NS, s_abort);
        }
        mail_phase ^= 1u;
        if (__syncthreads_or(fail)) timed_out = true;
        const int b = timed_out ? -2 : mail[level];
        if (timed_out) {
            if (tid == 0) cluster_drain(rank, C, smem_u32(s_abort), mbS, DRAIN_LIMIT_NS, DRAIN_GRACE_NS);
            __syncthreads();
            leave();
            return;
        }
        if (b < 0) {
            if (b == -2 || !P.split || G == 1) break;
            G /= 2;  // this class is exhausted: two groups from here on
            if (rank - g0 >= G) g0 += G;
            ++level;
            mail_phase = 0;
            continue;
        }

        int k0, Nb;
        P.bv.range(b, k0, Nb);
        const int c0 = k0 - b;  // first control/off-diagonal index
        const int KPC = ceil_div(Nb, G);
        const int kfirst = gr * KPC;  // instance-local index of slot 0
        const int k = kfirst + kl;    // this thread's knot
        const bool slot_knot = kl < KPC;  // knot slot in use (may lie past the horizon)
        const bool active_knot = slot_knot && k < Nb;
        const int max_iter = P.max_iter > 0 ? P.max_iter : 10 * Nb * NXR;
        // the warps holding the first and last knot slot (warp-uniform)
        const bool warp_left = has_left && warp == 0;
        const bool warp_right = has_right && warp == ((KPC - 1) * LPR) / 32;
        const uint32_t halo_bytes = (uint32_t)(NXR * sizeof(float)) * ((has_left ? 1u : 0u) + (has_right ? 1u : 0u));
        const bool rows = li < NXR / 2;               // lane 7 of a knot holds none
        const bool rv = active_knot && rows, st = slot_knot && rows;
        const int own = (kl + 1) * VSR + 2 * li;      // this thread's rows in a shared vector
        // A boundary knot's lanes keep the neighbour's halo copies current and
        // push their own rows: `side` is the side they face (a group with one
        // knot slot per CTA faces both: its left lanes repeat for the right).
        const bool hleft = kl == 0 && has_left && rows, hright = kl == KPC - 1 && has_right && rows;
        const bool hany = hleft || hright, hboth = hleft && hright;
        const int side = hleft ? 0 : 1, hbase = (side ? (KPC + 1) * VSR : 0) + 2 * li;
        const uint32_t nb = map_rank(smem_u32(smem), hleft ? rank - 1 : (hright ? rank + 1 : rank));
        const uint32_t nb_halo = nb + (uint32_t)(L.halo + sizeof(float) * ((1 - side) * VSR + 2 * li));
        const uint32_t nb_mbar = nb + (uint32_t)L.mbar;

        // ---- rows of S+ and Phi^-1 into registers -----------------------------
        float sd[2][NXR], sl[2][NXR], su[2][NXR];
        constexpr int NQ = PS ? 1 : NXR;
        float qd[2][NQ], ql[2][NQ], qu[2][NQ];  // (PS: in shared memory)
        float4 *mq = reinterpret_cast<float4 *>(smem + L.mats) + tid;
        {
            // Phi^-1 rows without off-diagonal blocks: every row for block
            // Jacobi (precon 1), the even knots' rows for the stair (2)
            const bool jac = P.precon == 1 || (P.precon == 2 && (k & 1) == 0);
            const bool hl = active_knot && k >= 1, hu = active_knot && k + 1 < Nb;
            const int n2 = NXR * NXR;
            const float *Sd = P.Sd + (size_t)(k0 + k) * n2, *Pd = P.Pd + (size_t)(k0 + k) * n2;
            const float *SoL = P.So + (ptrdiff_t)(c0 + k - 1) * n2, *PoL = P.Po + (ptrdiff_t)(c0 + k - 1) * n2;
            const float *SoU = P.So + (size_t)(c0 + k) * n2, *PoU = P.Po + (size_t)(c0 + k) * n2;
            // rows 2 li, 2 li + 1 of a block: down its columns (the diagonal
            // blocks are symmetric), or along its rows
            auto rows_of = [&](const float *M, bool on, bool along, auto &out) {
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int j = 0; j < NXR; ++j) {
                        const int i = 2 * li + m;
                        out[m][j] = on && rv ? __ldg(M + (along ? i * NXR + j : j * NXR + i)) : 0.f;
                    }
            };
            rows_of(Sd, true, false, sd);
            rows_of(SoL, hl, true, sl);
            rows_of(SoU, hu, false, su);
            if constexpr (PS) {
                auto stash = [&](int b, const float (&x)[2][NXR]) {
#pragma unroll
                    for (int q = 0; q < 3; ++q)
#pragma unroll
                        for (int m = 0; m < 2; ++m)
                            mq[(7 * b + 2 * q + m) * nthreads] = make_float4(x[m][4 * q], x[m][4 * q + 1], x[m][4 * q + 2], x[m][4 * q + 3]);
                    mq[(7 * b + 6) * nthreads] = make_float4(x[0][12], x[0][13], x[1][12], x[1][13]);
                };
                float x[2][NXR];
                rows_of(Pd, true, false, x);
                stash(0, x);
                rows_of(PoL, hl && !jac, true, x);
                stash(1, x);
                rows_of(PoU, hu && !jac, false, x);
                stash(2, x);
            } else {
                rows_of(Pd, true, false, qd);
                rows_of(PoL, hl && !jac, true, ql);
                rows_of(PoU, hu && !jac, false, qu);
            }
        }

        // Boundary rows into the neighbours' halo slots of vector v, one 8-byte
        // push per lane; bar: byte offset of the mbarrier among the CTA's.
        auto push_halo = [&](int v, uint32_t par, uint32_t bar, const float (&val)[2]) {
            if (!hany) return;
            const uint32_t off = (uint32_t)sizeof(float) * (uint32_t)halo_off(v, par, 0);
            st_async(nb_halo + off, dfloat{val[0], val[1]}, nb_mbar + bar);
            if (hboth) {
                const uint32_t nr = map_rank(smem_u32(smem), rank + 1);
                st_async(nr + (uint32_t)(L.halo + sizeof(float) * 2 * li) + off, dfloat{val[0], val[1]},
                         nr + (uint32_t)L.mbar + bar);
            }
        };

        // One thread, some way ahead of the exchange: the bytes that complete
        // it, with nh halo vectors travelling along.
        auto expect = [&](uint32_t nh) {
            if (G > 1 && tid == arm) mbar_arrive_expect(mb + 8 * (xr & 1u), (uint32_t)G * 32u + nh * halo_bytes);
        };
        // Group sums of four accumulators per thread.  Within a warp the four sums are reduced
        // by recursive halving (each lane gives away half of its sums per
        // level, 12 shuffles in place of 40); lanes 8u hold sum u.  The other
        // warps arrive on named barrier 1 and go on to wait; warp 0 waits
        // there, adds the warp sums and pushes them in pairs, lanes 0-15 sums
        // 0 and 1 to CTA lane, lanes 16-31 sums 2 and 3 to CTA lane - 16.
        auto exchange = [&](A v0, A v1, A v2, A v3) -> Sums {
            const uint32_t par = xr & 1u, bar = mb + 8 * par;
            const bool h16 = lane & 16, h8 = lane & 8;
            A a = AT::add_tree(h16 ? v2 : v0, AT::shfl_xor(h16 ? v0 : v2, 16));
            A c = AT::add_tree(h16 ? v3 : v1, AT::shfl_xor(h16 ? v1 : v3, 16));
            A x = AT::add_tree(h8 ? c : a, AT::shfl_xor(h8 ? a : c, 8));
#pragma unroll
            for (int m = 4; m >= 1; m >>= 1) x = AT::add_tree(x, AT::shfl_xor(x, m));
            const int u = lane >> 3, w8 = lane & 7;
            if (w8 == 0) wpart[(u >> 1) * 2 * WMAX + 2 * warp + (u & 1)] = x;
            if (G == 1) {  // no peers: every warp adds the warp sums
                __syncthreads();
                x = wpart[(u >> 1) * 2 * WMAX + 2 * w8 + (u & 1)];
#pragma unroll
                for (int m = 4; m >= 1; m >>= 1) x = AT::add_tree(x, AT::shfl_xor(x, m));
            } else {
                const int q = lane & 15, pr = lane >> 4;
                const uint32_t slot_off = (uint32_t)((((int)par * 2 + pr) * CMAX) * 16);
                if (warp == 0) {
                    const uint32_t pb = map_rank(smem_u32(smem), g0 + (q < G ? q : 0));
                    named_bar_sync(1, nthreads);
                    // every wpow lanes load the W warp sums of their pair
                    // (those of absent warps are zero)
                    A y0, y1;
                    load_pair(wpart + pr * 2 * WMAX + 2 * (lane & (wpow - 1)), y0, y1);
                    auto level = [&](int m) {
                        y0 = AT::add_tree(y0, AT::shfl_xor(y0, m));
                        y1 = AT::add_tree(y1, AT::shfl_xor(y1, m));
                    };
                    if (W > 4) level(4);
                    if (W > 2) level(2);
                    if (W > 1) level(1);
                    if (q < G)
                        push_pair(pb + (uint32_t)L.slot + slot_off + 16u * (uint32_t)gr, y0, y1, pb + (uint32_t)L.mbar + 8 * par);
                } else {
                    named_bar_arrive(1, nthreads);
                }
                // one warp polls, a CTA barrier wakes the others
                if (warp == 0 && warp_wait(bar, (xr >> 1) & 1u, s_abort)) *s_fail = 1;
                __syncthreads();
                A p0 = AT::zero(), p1 = AT::zero();
                if (q < G) load_pair(reinterpret_cast<const A *>(slots + slot_off + 16 * q), p0, p1);
                x = AT::add_tree(h8 ? p1 : p0, AT::shfl_xor(h8 ? p0 : p1, 8));
#pragma unroll
                for (int m = 4; m >= 1; m >>= 1) x = AT::add_tree(x, AT::shfl_xor(x, m));
            }
            ++xr;
            Sums r;
            const float xf = AT::to_T(x);
            r.eta = bcast(x, 0);
            r.rr = __shfl_sync(0xffffffffu, xf, 8);
            r.del = __shfl_sync(0xffffffffu, xf, 16);
            r.eps = __shfl_sync(0xffffffffu, xf, 24);
            return r;
        };

        // ---- initialisation: r = b - S lambda0, ||b||^2 ---------------------------
        for (int e = tid; e < (P.kpc_max + 2) * VSR; e += nthreads) vecR[e] = vecP[e] = vecZ[e] = 0.f;
        __syncthreads();
        float lam[2] = {0.f, 0.f}, r[2] = {0.f, 0.f}, p[2] = {0.f, 0.f}, s[2] = {0.f, 0.f};
        const bool mode1 = P.tol_mode == 1;
        float tol_t;
        A bb;
        {
            float bv[2] = {0.f, 0.f};
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int i = 2 * li + m;
                if (rv) {
                    lam[m] = P.lam[(size_t)(k0 + k) * NXR + i];
                    bv[m] = P.rhs_sign * P.rhs[(size_t)(k0 + k) * NXR + i];
                    vecZ[own + m] = lam[m];
                }
                // lambda0 halo straight from global memory
                if (rows && kl == 0 && kfirst >= 1 && kfirst - 1 < Nb) vecZ[i] = P.lam[(size_t)(k0 + kfirst - 1) * NXR + i];
                if (rows && kl == KPC - 1 && kfirst + KPC < Nb)
                    vecZ[(KPC + 1) * VSR + i] = P.lam[(size_t)(k0 + kfirst + KPC) * NXR + i];
            }
            __syncthreads();
            const float *vp = vecZ + kl * VSR;
            if (rv) {
                r[0] = resid_row(bv[0], sd[0], sl[0], su[0], vp, vp + VSR, vp + 2 * VSR);
                r[1] = resid_row(bv[1], sd[1], sl[1], su[1], vp, vp + VSR, vp + 2 * VSR);
            }
            if (st) *reinterpret_cast<float2 *>(vecR + own) = make_float2(r[0], r[1]);
            const uint32_t par = xr & 1u;
            push_halo(1, par, 8 * par, r);
            expect(1u);
            bb = exchange(AT::add(AT::prod(bv[0], bv[0]), AT::prod(bv[1], bv[1])), AT::zero(), AT::zero(), AT::zero()).eta;
            if (hany) *reinterpret_cast<float2 *>(vecR + hbase) = *reinterpret_cast<const float2 *>(halo + halo_off(1, par, side) + 2 * li);
            if (hboth)
                *reinterpret_cast<float2 *>(vecR + 2 * VSR + 2 * li) = *reinterpret_cast<const float2 *>(halo + halo_off(1, par, 1) + 2 * li);
            const double tol = P.tol > 0 ? P.tol : 1e-6;
            tol_t = mode1 ? (float)tol : (float)(tol * tol * AT::to_double(bb));
        }
        __syncthreads();

        // Scalars of the iteration (alpha, beta, exit tests) are taken in
        // float from the extended sums.
        A eta = AT::zero();
        float ups = 0.f, inv_eta = 0.f, rr = 0.f;
        int iters = 0;
        bool broke = false;
        int it = 0;
        for (;; ++it) {
            // ---- r~ = Phi^-1 r, boundary rows to the neighbours -----------------
            const uint32_t zpar = xz & 1u, rpar = xr & 1u;  // halo rows alternate once per iteration
            const int failed = *s_fail;  // before the barrier: as every warp saw it
            float z[2] = {0.f, 0.f}, q[2] = {0.f, 0.f}, t[2] = {0.f, 0.f};
            if (active_knot) {
                const float *vp = vecR + kl * VSR;
                if constexpr (PS) rowdot2_ps(mq, nthreads, vp, vp + VSR, vp + 2 * VSR, z);
                else rowdot2(qd, ql, qu, vp, vp + VSR, vp + 2 * VSR, z);
            }
            push_halo(0, zpar, 16, z);
            if (st) *reinterpret_cast<float2 *>(vecZ + own) = make_float2(z[0], z[1]);
            if (G > 1 && tid == arm) mbar_arrive_expect(mbZ, halo_bytes);
            expect(2u);
            // ---- S p_old and the sums without S r~, while they travel -------------
            if (active_knot) {
                const float *vp = vecP + kl * VSR;
                rowdot2(sd, sl, su, vp, vp + VSR, vp + 2 * VSR, t);
            }
            push_halo(2, zpar, 8 * rpar, t);
            const A s_eta = AT::add(AT::prod(r[0], z[0]), AT::prod(r[1], z[1]));
            const A s_rr = sq_sum(r[0], r[1], A{});
            const A s_eps = AT::add(AT::prod(z[0], s[0]), AT::prod(z[1], s[1]));
            if (failed) {
                timed_out = true;
                break;
            }
            __syncthreads();
            // ---- S r~ ------------------------------------------------------------
            if (warp_left || warp_right)
                if (warp_wait(mbZ, xz & 1u, s_abort)) *s_fail = 1;
            ++xz;
            if (active_knot) {
                const float *vp = vecZ + kl * VSR;
                rowdot2(sd, sl, su, kl == 0 && has_left ? halo + halo_off(0, zpar, 0) : vp, vp + VSR,
                        kl == KPC - 1 && has_right ? halo + halo_off(0, zpar, 1) : vp + 2 * VSR, q);
            }
            push_halo(1, zpar, 8 * rpar, q);
            // the boundary lanes' halo operands are loaded before alpha and beta are formed
            float2 hz, hq, ht, hp, hr;
            hz = hq = ht = hp = hr = make_float2(0.f, 0.f);
            const float *hsrc = halo + halo_off(0, 0, side) + 2 * li;
            if (hany) {
                hz = *reinterpret_cast<const float2 *>(hsrc + halo_off(0, zpar, 0));
                hp = *reinterpret_cast<const float2 *>(vecP + hbase);
                hr = *reinterpret_cast<const float2 *>(vecR + hbase);
            }
            const Sums S = exchange(s_eta, s_rr, AT::add(AT::prod(z[0], q[0]), AT::prod(z[1], q[1])), s_eps);
            if (hany) {
                hq = *reinterpret_cast<const float2 *>(hsrc + halo_off(1, zpar, 0));
                ht = *reinterpret_cast<const float2 *>(hsrc + halo_off(2, zpar, 0));
            }
            eta = S.eta;
            rr = S.rr;
            const float etan = AT::to_T(S.eta);
            const float beta = __fmul_rn(etan, inv_eta);  // 0 in the first iteration
            ups = __fmaf_rn(beta, __fmaf_rn(beta, ups, S.eps + S.eps), S.del);
            float alpha = __fdividef(etan, ups);
            const bool done = !(fabsf(etan) <= 3.402823466e38f && rr <= 3.402823466e38f) ||
                              (mode1 ? etan < tol_t : rr <= tol_t) || it >= max_iter;
            // the identity cancelled, or S+ is not positive on p (or not finite)
            const bool direct = !(ups > 0.0625f * S.del && ups <= 3.402823466e38f);
            // p = r~ + beta p, S p = S r~ + beta S p_old, lambda += alpha p,
            // r -= alpha S p; the halo copies of p and r alike
            auto next_p = [&]() {
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    s[m] = fma_rn(beta, t[m], q[m]);
                    p[m] = fma_rn(beta, p[m], z[m]);
                }
            };
            auto apply = [&]() {
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    r[m] = fma_rn(-alpha, s[m], r[m]);
                    lam[m] = fma_rn(alpha, p[m], lam[m]);
                }
                if (st) {
                    *reinterpret_cast<float2 *>(vecR + own) = make_float2(r[0], r[1]);
                    *reinterpret_cast<float2 *>(vecP + own) = make_float2(p[0], p[1]);
                }
                if (hany) {
                    *reinterpret_cast<float2 *>(vecR + hbase) = make_float2(fma_rn(-alpha, fma_rn(beta, ht.x, hq.x), hr.x),
                                                                            fma_rn(-alpha, fma_rn(beta, ht.y, hq.y), hr.y));
                    *reinterpret_cast<float2 *>(vecP + hbase) = make_float2(fma_rn(beta, hp.x, hz.x), fma_rn(beta, hp.y, hz.y));
                }
                if (hboth) {
                    const float *h = halo + halo_off(0, 0, 1) + 2 * li;
                    for (int m = 0; m < 2; ++m) {
                        float *vr = vecR + 2 * VSR + 2 * li + m, *vp = vecP + 2 * VSR + 2 * li + m;
                        *vr = fma_rn(-alpha, fma_rn(beta, h[halo_off(2, zpar, 0) + m], h[halo_off(1, zpar, 0) + m]), *vr);
                        *vp = fma_rn(beta, *vp, h[halo_off(0, zpar, 0) + m]);
                    }
                }
            };
            if (!done) {
                next_p();
                if (!direct) apply();
            }
            inv_eta = __fdividef(1.f, etan);
            iters = it;
            __syncthreads();
            if (done || direct) {
                // a warp that gave up its wait may have come to another
                // decision: it leaves at its next check, the others here
                if (*s_fail) {
                    timed_out = true;
                    break;
                }
                if (done) break;
                // sum p^T S p itself
                expect(0u);
                ups = AT::to_T(exchange(AT::add(AT::prod(p[0], s[0]), AT::prod(p[1], s[1])), AT::zero(), AT::zero(), AT::zero()).eta);
                if (!(ups > 0.f) || !isfinite(ups)) {
                    broke = true;
                    iters = it + 1;
                } else {
                    alpha = AT::div(etan, ups);
                    apply();
                }
                __syncthreads();
                if (*s_fail) timed_out = true;
                if (broke || timed_out) break;
            }
        }
        // ---- write back ----------------------------------------------------------
        if (rv)
            for (int m = 0; m < 2; ++m) P.lam[(size_t)(k0 + k) * NXR + 2 * li + m] = lam[m];
        if (gr == 0 && tid == 0 && P.stats) {
            const float etan = AT::to_T(eta);
            mpcg_stats st;
            st.iters = iters;
            st.status = timed_out ? MPCG_TIMEOUT
                        : broke   ? MPCG_BREAKDOWN
                        : !(isfinite(etan) && isfinite(rr))         ? MPCG_NONFINITE
                        : (mode1 ? etan < tol_t : rr <= tol_t)      ? MPCG_CONVERGED
                                                                    : MPCG_NOT_CONVERGED;
            st.eta = AT::to_double(eta);
            const double bbd = AT::to_double(bb), rrd = (double)rr;
            st.relres = bbd > 0.0 ? sqrt(rrd / bbd) : sqrt(rrd);
            P.stats[b] = st;
        }
        // A CTA whose wait gave up (or that a peer told to stop) must not
        // enter another cluster-wide barrier, which a stuck peer would never
        // reach, nor leave while peers may still push into its shared memory:
        // it drains the cluster (cluster_drain) and leaves.
        if (timed_out) {
            if (tid == 0) cluster_drain(rank, C, smem_u32(s_abort), mbS, DRAIN_LIMIT_NS, DRAIN_GRACE_NS);
            __syncthreads();
            leave();
            return;
        }
        // No barrier between instances: a peer that is already at the next
        // one pushes into the other parity's buffers, and can get no further
        // before this CTA's sums for it arrive.
    }
    cluster_sync_all();  // peers may push into this CTA's shared memory until they leave too
    leave();
}

size_t pcg_reg_smem_bytes(const PcgLaunch &L) { return RegLayout(L.kpc_max, L.reg == 2 ? L.threads : 0).total; }

static void (*reg_fn(const PcgLaunch &L))(const PcgParams<float>) {
    if (L.reg == 2) return L.dot ? pcg_reg_kernel<AccF64, true> : pcg_reg_kernel<Acc<float>, true>;
    return L.dot ? pcg_reg_kernel<AccF64, false> : pcg_reg_kernel<Acc<float>, false>;
}

static cudaLaunchConfig_t reg_config(const PcgLaunch &L, int clusters, cudaLaunchAttribute *attr, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.C * clusters, 1, 1);
    cfg.blockDim = dim3(L.threads, 1, 1);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = L.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

cudaError_t pcg_reg_launch(const PcgLaunch &L, const PcgParams<float> &P0, cudaStream_t s) {
    PcgParams<float> P = P0;
    P.kpc_max = L.kpc_max;
    P.vs = VSR;
    cudaLaunchAttribute attr[2];
    PcgLaunch S = L;
    P.n_upto = INT_MAX;
    int full = 1;  // sizes of the stages: full, 3/4 full, 1/2 full
    while (full < L.C) full *= 2;
    const int mid = 3 * full / 4, low = full / 2;
    for (int stage = 0;; ++stage) {
        const bool to_mid = P.queue && L.n_mid > 0 && S.C > mid, to_low = P.queue && L.n_mid > 0 && S.C == mid;
        P.n_above = to_mid ? mid * L.kpc_max : to_low ? low * L.kpc_max : INT_MIN;
        P.split = to_mid || to_low ? 0 : L.split;
        cudaLaunchConfig_t cfg = reg_config(S, S.clusters, attr, s);
        if (stage) cfg.numAttrs = 2;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, reg_fn(S), P);
        if (e != cudaSuccess || !(to_mid || to_low)) return e;
        P.n_upto = P.n_above;
        P.queue += QUEUE_LEVELS;
        S.C = to_mid ? mid : low;
        S.clusters = to_mid ? L.n_mid : L.n_low;
    }
}

int pcg_reg_max_clusters(const PcgLaunch &L) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = reg_config(L, 1, attr, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, reg_fn(L), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t pcg_reg_prepare(int smem_optin) {
    for (auto *fn : {pcg_reg_kernel<Acc<float>, false>, pcg_reg_kernel<AccF64, false>, pcg_reg_kernel<Acc<float>, true>,
                     pcg_reg_kernel<AccF64, true>}) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace mpcg
