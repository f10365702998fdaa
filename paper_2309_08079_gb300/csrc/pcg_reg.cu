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
// nor symmetry of Phi^-1).  S p = S r~ + beta S p_old takes S p_old from a
// fresh product of the stored p each iteration; p_old^T S p_old is carried, in
// float pairs, with most of it taken anew in each iteration (curvature in
// pcg_sums.cuh).  Emulated in float32 on the Kuka-shaped problems
// (N = 32..512, cold and warm), iteration counts equal Algorithm 1's and
// lambda differs from it by what another summation order changes (1e-6 warm).
// The Chronopoulos-Gear form, which carries S p by recurrence, is 3 to 10
// times further off.  The price is a third product, 84 FMAs per lane, which
// runs while the boundary rows of r~ travel to the neighbour CTAs.  Where the
// identity cancels (p^T S p below about 1/32 of its terms; 0.29 of r~^T S r~ was the
// smallest share seen on the emulated problems) or too much of the carried
// error is passed on, the sum p^T S p is taken directly with one more
// reduction.  Measured on GB300 at fixed iteration counts: 1.83 us per
// iteration at N = 512 (16 CTAs x 32 knots) and 1.57 at N = 128 (16 x 8) against
// 2.23 and 1.98 with two reductions.  Of the 1.83 us, by leaving parts out one
// at a time: the three products 0.2-0.3 each (bound by the shared-memory reads
// of the vectors, 128 bytes per clock), the warp sums 0.11, the CTA sums 0.11,
// the sums over CTAs 0.06, p^T S p in float pairs 0.06; the rest is the transport
// (0.12 one way) and the CTA barriers.
//
// Launch shape: clusters of C <= 16 CTAs; a group of G CTAs (the whole
// cluster, or a power-of-two part of it, below) solves one instance; CTA r of
// the group owns knots [r KPC, (r+1) KPC), KPC = ceil(N/G) <= 32; 8 lanes own
// a knot, lanes 0..6 two adjacent rows each, and keep their rows of S+ and
// Phi^-1 (2 x 84 floats) in registers for the whole solve.  r, p, r~ (with
// one halo knot on each side) live in shared memory.
//
// PS form, for batches: with many instances the exchanges of one leave the SM
// idle two thirds of the time.  Four lanes own a knot, four rows each, their rows
// of S+ (168 floats) in registers and those of Phi^-1 in shared memory, so a CTA of
// 32 knots has 128 threads and two share an SM.  (A lane's vector loads serve
// four rows: half the shared-memory reads of vectors that bound the form it
// replaces, 8 lanes and 128 registers.)  An iteration takes 1.7-1.8 times as
// long as alone.  Up to 64 knots one CTA of 256 threads holds an instance, without
// exchanges (256 of 60..64 knots 1.07 against 1.22 ms); longer ones are better in
// CTAs of 32 knots, which overlap (64 of 128 knots 1.17 against 1.24 with 64).
// Former form -> this one: 256 instances of 32..512 knots 19.9 -> 16.5 ms, 256 of
// 60..64 1.48 -> 1.05, 150 of 100..250 5.85 -> 4.9, 17 of 505..512 3.97 -> 3.8.
// (These times, and those below, are of a p^T S p in plain float; in pairs batches
// take 3 to 5 % more: 17.1, 1.10, 5.05 and 4.0 ms.)
//
// Choice of the form: PS pays once the other would need a second wave; that
// depends on the horizons, which the host does not know.  Between one and four
// waves by count both forms are launched, and each CTA sums CTAs x knots over the
// instances (the time of a wave): above 0.95 of one wave of the longest horizon the
// PS launches do the work, below it the others, and the rest leave at once (5 to 20
// us).  Register form / PS / chosen: 60 instances of 20..128 knots 0.68 / 0.98 /
// 0.69 ms, 25 of 40..256 1.07 / 1.63 / 1.07, 64 of 128 1.37 / 1.17 / 1.19, 9 of 512
// 2.63 / 2.07-2.20 / 2.20, 200 of 16..32 0.285 / 0.291 / 0.315.
//
// Groups: a launch with more instances than clusters splits its clusters as
// the long instances run out.  At level l a group of C >> l CTAs takes only
// instances that need more than half of it at 32 knots per CTA; when that
// class is exhausted the group splits in two.  A ragged batch then runs its
// long horizons first, and short ones do not occupy a whole cluster (256
// instances of 32..512 knots: 42.8 ms with a 16-CTA cluster for each and two
// reductions, 27.5 ms split).
//
// Stages: a GPC holds one or two clusters of 16 and then has SMs to spare (14
// clusters, 224 of 304 CTAs, with two CTAs per SM), and 257..384 knots need no
// 16.  So a batch of more than one wave takes up to three launches, for the
// horizons that need full clusters (16, 8 or 4 CTAs), those that 3/4 hold and those
// that half holds (which split); each may begin in the SMs that the one before
// leaves free.  One launch -> stages (with the former PS form): 256 instances of 32..512 knots 25.5 -> 19.9
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
// Floats per knot slot of a shared vector (16 used): 20 puts the 16-byte words
// of eight consecutive knots, one load of the PS form, on distinct banks (16: 22 %
// of its shared-memory wavefronts were conflicts; 64 instances of 128 knots 1.21
// against 1.12 ms, 256 of 60..64 1.08 against 1.05).
constexpr int VSR = 20;
constexpr int CMAX = 16;  // CTAs per cluster
constexpr int WMAX = 8;   // warps per CTA
constexpr int LEVELS = 5; // group sizes C, C/2, ..., C/16

// Shared-memory carve-up, in bytes; the same on host and device.
struct RegLayout {
    size_t vecR, vecP, vecZ, halo, slot, wpart, mbar, mail, misc, mats, total;
    // threads > 0: the rows of Phi^-1 of so many threads too, four each
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
        mats = take(sizeof(float) * (size_t)(3 * 4 * NXR) * threads);
        total = o;
    }
};

// R rows of one block row times the halo'd vector: the knot's three
// vector slots are read once for all of them.
template <int R>
__device__ __forceinline__ void rowdot(const float (&d)[R][NXR], const float (&l)[R][NXR], const float (&u)[R][NXR],
                                       const float *vprev, const float *vself, const float *vnext, float (&y)[R]) {
    float a0[R], a1[R], a2[R];
#pragma unroll
    for (int m = 0; m < R; ++m) a0[m] = a1[m] = a2[m] = 0.f;
    const float4 *p4 = reinterpret_cast<const float4 *>(vprev);
    const float4 *s4 = reinterpret_cast<const float4 *>(vself);
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
#pragma unroll
                for (int m = 0; m < R; ++m) a0[m] = __fmaf_rn(d[m][j], vs_[t], a0[m]);
#pragma unroll
                for (int m = 0; m < R; ++m) a1[m] = __fmaf_rn(l[m][j], vp_[t], a1[m]);
#pragma unroll
                for (int m = 0; m < R; ++m) a2[m] = __fmaf_rn(u[m][j], vn_[t], a2[m]);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < R; ++m) y[m] = (a0[m] + a1[m]) + a2[m];
}

// The same with the thread's four rows in shared memory (PS form): 42
// four-entry words per thread, word c of all threads side by side, so a warp's
// load is conflict-free; per block 14 words, the rows' entries 4 q .. 4 q + 3 in
// turn (the last two: entries 12 and 13 of two rows each).
__device__ __forceinline__ void rowdot_ps(const float4 *m, int stride, const float *v, float (&y)[4]) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {  // diagonal, lower, upper
        const float4 *v4 = reinterpret_cast<const float4 *>(v + (b == 0 ? VSR : b == 1 ? 0 : 2 * VSR));
        const float4 *w = m + (size_t)14 * b * stride;
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 x = v4[q];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 e = w[(4 * q + i) * stride];
                a[i] = __fmaf_rn(e.x, x.x, a[i]);
                a[i] = __fmaf_rn(e.y, x.y, a[i]);
                a[i] = __fmaf_rn(e.z, x.z, a[i]);
                a[i] = __fmaf_rn(e.w, x.w, a[i]);
            }
        }
        const float2 x = *reinterpret_cast<const float2 *>(v4 + 3);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 e = w[(12 + h) * stride];
            a[2 * h] = __fmaf_rn(e.y, x.y, __fmaf_rn(e.x, x.x, a[2 * h]));
            a[2 * h + 1] = __fmaf_rn(e.w, x.y, __fmaf_rn(e.z, x.x, a[2 * h + 1]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = b == 0 ? a[i] : y[i] + a[i];
    }
}

// a thread's rows as one word of a shared vector
__device__ __forceinline__ void put(float *p, const float (&v)[2]) { *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]); }
__device__ __forceinline__ void put(float *p, const float (&v)[4]) { *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void get(const float *p, float (&v)[2]) {
    const float2 x = *reinterpret_cast<const float2 *>(p);
    v[0] = x.x; v[1] = x.y;
}
__device__ __forceinline__ void get(const float *p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4 *>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void push_rows(uint32_t a, const float (&v)[2], uint32_t mbar) { st_async(a, dfloat{v[0], v[1]}, mbar); }
__device__ __forceinline__ void push_rows(uint32_t a, const float (&v)[4], uint32_t mbar) { st_async_v4(a, v[0], v[1], v[2], v[3], mbar); }

__device__ __forceinline__ float resid_row(float b, const float (&d)[NXR], const float (&l)[NXR],
                                           const float (&u)[NXR], const float *v) {
    dfloat a{b, 0.f};
#pragma unroll
    for (int j = 0; j < NXR; ++j) {
        a = df_add(a, df_prod(-d[j], v[VSR + j]));
        a = df_add(a, df_prod(-l[j], v[j]));
        a = df_add(a, df_prod(-u[j], v[2 * VSR + j]));
    }
    return __fadd_rn(a.hi, a.lo);
}

}  // namespace

template <typename AT, bool PS>
__global__ void __launch_bounds__(32 * WMAX, 1) pcg_reg_kernel(const PcgParams<float> P) {
    using A = typename AT::type;
    static_assert(sizeof(A) == 8, "sums travel in pairs of 8 bytes");
    extern __shared__ __align__(16) unsigned char smem[];
    struct Sums {
        A eta, del, eps;  // r^T r~, r~^T S r~, (r~ + g / 2 p_old)^T S p_old
        float rr;         // ||r||^2
    };

    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int nthreads = blockDim.x, W = nthreads / 32;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    constexpr int R = PS ? 4 : 2, LPR = 16 / R;  // rows per lane, lanes per knot
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

    grid_dep_launch();
    // the next stage overlaps this one, so the last must outlive them all: one
    // thread of each stage leaves only when the stage before it is complete
    auto leave = [&]() {
        if (blockIdx.x == 0 && tid == 0) grid_dep_wait();
    };

    if (P.pick) {  // is this form the batch's? (every CTA of both forms finds the same)
        unsigned long long *sum = reinterpret_cast<unsigned long long *>(wpart), w = 0;
        if (tid == 0) *sum = 0;
        __syncthreads();
        for (int t = tid; t < P.n_tickets; t += nthreads) {
            int k0, Nb;
            P.bv.range(P.inst_list ? P.inst_list[t] : t, k0, Nb);
            if (Nb < 1 || Nb > P.n_long) continue;
            int need = 1;
            while (32 * need < Nb) need *= 2;
            if (need >= 4 && 24 * need >= Nb) need -= need / 4;
            w += (unsigned long long)need * Nb;
        }
        for (int m = 16; m >= 1; m >>= 1) w += __shfl_xor_sync(0xffffffffu, w, m);
        if (lane == 0) atomicAdd(sum, w);
        __syncthreads();
        const bool heavy = (long long)*sum > P.work;
        __syncthreads();  // wpart is cleared below
        if (heavy != (P.pick > 0)) {
            leave();
            return;
        }
    }
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
                if (b < 0) break;  // ends this pass over the list for the group, as its end does
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
        const int b = mail[level];
        if (timed_out) {
            if (tid == 0) cluster_drain(rank, C, smem_u32(s_abort), mbS, DRAIN_LIMIT_NS, DRAIN_GRACE_NS);
            __syncthreads();
            leave();
            return;
        }
        if (b < 0) {
            if (!P.split || G == 1) break;
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
        const uint32_t halo_bytes = (uint32_t)((PS ? 16 : NXR) * sizeof(float)) * ((has_left ? 1u : 0u) + (has_right ? 1u : 0u));
        const bool rows = R * li < NXR;               // (R = 2) lane 7 of a knot holds none
        const bool rv = active_knot && rows, st = slot_knot && rows;
        const int own = (kl + 1) * VSR + R * li;      // this thread's rows in a shared vector
        // A boundary knot's lanes keep the neighbour's halo copies current and
        // push their own rows: `side` is the side they face (a group with one
        // knot slot per CTA faces both: its left lanes repeat for the right).
        const bool hleft = kl == 0 && has_left && rows, hright = kl == KPC - 1 && has_right && rows;
        const bool hany = hleft || hright, hboth = hleft && hright;
        const int side = hleft ? 0 : 1, hbase = (side ? (KPC + 1) * VSR : 0) + R * li;
        const uint32_t nb = map_rank(smem_u32(smem), hleft ? rank - 1 : (hright ? rank + 1 : rank));
        const uint32_t nb_halo = nb + (uint32_t)(L.halo + sizeof(float) * ((1 - side) * VSR + R * li));
        const uint32_t nb_mbar = nb + (uint32_t)L.mbar;

        // ---- rows of S+ and Phi^-1 into registers -----------------------------
        float sd[R][NXR], sl[R][NXR], su[R][NXR];
        constexpr int NQ = PS ? 1 : NXR;
        float qd[R][NQ], ql[R][NQ], qu[R][NQ];  // (PS: in shared memory)
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
            // rows R li .. of a block (none past the last): down its columns (the diagonal
            // blocks are symmetric), or along its rows
            auto rows_of = [&](const float *M, bool on, bool along, auto &out) {
#pragma unroll
                for (int m = 0; m < R; ++m)
#pragma unroll
                    for (int j = 0; j < NXR; ++j) {
                        const int i = R * li + m;
                        out[m][j] = on && rv && (NXR % R == 0 || i < NXR) ? __ldg(M + (along ? i * NXR + j : j * NXR + i)) : 0.f;
                    }
            };
            rows_of(Sd, true, false, sd);
            rows_of(SoL, hl, true, sl);
            rows_of(SoU, hu, false, su);
            if constexpr (PS) {
                auto stash = [&](int b, const float (&x)[R][NXR]) {
#pragma unroll
                    for (int q = 0; q < 3; ++q)
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            mq[(14 * b + 4 * q + m) * nthreads] = make_float4(x[m][4 * q], x[m][4 * q + 1], x[m][4 * q + 2], x[m][4 * q + 3]);
                    for (int h = 0; h < 2; ++h)
                        mq[(14 * b + 12 + h) * nthreads] = make_float4(x[2 * h][12], x[2 * h][13], x[2 * h + 1][12], x[2 * h + 1][13]);
                };
                float x[R][NXR];
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

        // Boundary rows into the neighbours' halo slots of vector v, one push
        // per lane; bar: byte offset of the mbarrier among the CTA's.
        auto push_halo = [&](int v, uint32_t par, uint32_t bar, const float (&val)[R]) {
            if (!hany) return;
            const uint32_t off = (uint32_t)sizeof(float) * (uint32_t)halo_off(v, par, 0);
            push_rows(nb_halo + off, val, nb_mbar + bar);
            if (hboth) {
                const uint32_t nr = map_rank(smem_u32(smem), rank + 1);
                push_rows(nr + (uint32_t)(L.halo + sizeof(float) * R * li) + off, val, nr + (uint32_t)L.mbar + bar);
            }
        };
        // x . y over this thread's rows
        auto dot = [](const float (&x)[R], const float (&y)[R]) -> A {
            A a = AT::add(AT::prod(x[0], y[0]), AT::prod(x[1], y[1]));
            if constexpr (R == 4) a = AT::add(a, AT::add(AT::prod(x[2], y[2]), AT::prod(x[3], y[3])));
            return a;
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
            r.del = bcast(x, 16);
            r.eps = bcast(x, 24);
            return r;
        };

        // ---- initialisation: r = b - S lambda0, ||b||^2 ---------------------------
        for (int e = tid; e < (P.kpc_max + 2) * VSR; e += nthreads) vecR[e] = vecP[e] = vecZ[e] = 0.f;
        __syncthreads();
        float lam[R] = {}, r[R] = {}, p[R] = {}, s[R] = {};
        const bool mode1 = P.tol_mode == 1;
        float tol_t;
        A bb;
        {
            float bv[R] = {};
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const int i = R * li + m;
                if (i >= NXR) continue;
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
#pragma unroll
                for (int m = 0; m < R; ++m) r[m] = resid_row(bv[m], sd[m], sl[m], su[m], vp);
            }
            if (st) put(vecR + own, r);
            const uint32_t par = xr & 1u;
            push_halo(1, par, 8 * par, r);
            expect(1u);
            bb = exchange(dot(bv, bv), AT::zero(), AT::zero(), AT::zero()).eta;
            float h[R];
            if (hany) {
                get(halo + halo_off(1, par, side) + R * li, h);
                put(vecR + hbase, h);
            }
            if (hboth) {
                get(halo + halo_off(1, par, 1) + R * li, h);
                put(vecR + 2 * VSR + R * li, h);
            }
            const double tol = P.tol > 0 ? P.tol : 1e-6;
            tol_t = mode1 ? (float)tol : (float)(tol * tol * AT::to_double(bb));
        }
        __syncthreads();

        // Scalars of the iteration (alpha, beta, exit tests) are taken in
        // float from the extended sums.
        A eta = AT::zero(), acc = AT::zero();  // acc: p^T S p
        float rr = 0.f, g = 0.f;  // g: the last beta
        EtaRecip<float> recip;
        int iters = 0;
        bool broke = false;
        int it = 0;
        for (;; ++it) {
            // ---- r~ = Phi^-1 r, boundary rows to the neighbours -----------------
            const uint32_t zpar = xz & 1u, rpar = xr & 1u;  // halo rows alternate once per iteration
            const int failed = *s_fail;  // before the barrier: as every warp saw it
            float z[R] = {}, q[R] = {}, t[R] = {};
            if (active_knot) {
                const float *vp = vecR + kl * VSR;
                if constexpr (PS) rowdot_ps(mq, nthreads, vp, z);
                else rowdot<R>(qd, ql, qu, vp, vp + VSR, vp + 2 * VSR, z);
            }
            push_halo(0, zpar, 16, z);
            if (st) put(vecZ + own, z);
            if (G > 1 && tid == arm) mbar_arrive_expect(mbZ, halo_bytes);
            expect(2u);
            // ---- S p_old and the sums without S r~, while they travel -------------
            if (active_knot) {
                const float *vp = vecP + kl * VSR;
                rowdot<R>(sd, sl, su, vp, vp + VSR, vp + 2 * VSR, t);
            }
            push_halo(2, zpar, 8 * rpar, t);
            const A s_eta = dot(r, z);
            A s_rr = sq_sum(r[0], r[1], A{});
            if constexpr (R == 4) s_rr = AT::add(s_rr, sq_sum(r[2], r[3], A{}));
            float w[R];
#pragma unroll
            for (int m = 0; m < R; ++m) w[m] = __fmaf_rn(0.5f * g, p[m], z[m]);
            const A s_eps = dot(w, s);
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
                rowdot<R>(sd, sl, su, kl == 0 && has_left ? halo + halo_off(0, zpar, 0) : vp, vp + VSR,
                          kl == KPC - 1 && has_right ? halo + halo_off(0, zpar, 1) : vp + 2 * VSR, q);
            }
            push_halo(1, zpar, 8 * rpar, q);
            // the boundary lanes' halo operands are loaded before alpha and beta
            // are formed (PS: when used, there are no registers to spare)
            constexpr int RH = PS ? 1 : R;
            float hz[RH], hq[RH], ht[RH], hp[RH], hr[RH];
            const float *hsrc = halo + halo_off(0, 0, side) + R * li;
            if constexpr (!PS) {
#pragma unroll
                for (int m = 0; m < R; ++m) hz[m] = hq[m] = ht[m] = hp[m] = hr[m] = 0.f;
                if (hany) {
                    get(hsrc + halo_off(0, zpar, 0), hz);
                    get(vecP + hbase, hp);
                    get(vecR + hbase, hr);
                }
            }
            const Sums S = exchange(s_eta, s_rr, dot(z, q), s_eps);
            if constexpr (!PS) {
                if (hany) {
                    get(hsrc + halo_off(1, zpar, 0), hq);
                    get(hsrc + halo_off(2, zpar, 0), ht);
                }
            }
            const float etan = AT::to_T(S.eta);
            const float beta = recip.beta(etan, 0.f);  // 0 in the first iteration
            eta = S.eta;
            rr = S.rr;
            const A old = acc;
            acc = curvature(S.del, S.eps, acc, beta, g);
            float ups = rounded(acc, 0.f), alpha = __fdividef(etan, ups);
            const bool done = !(fabsf(etan) <= 3.402823466e38f && rr <= 3.402823466e38f) ||
                              (mode1 ? etan < tol_t : rr <= tol_t) || it >= max_iter;
            const bool direct = doubtful(ups, S.del, S.eps, old, beta, g);
            // p = r~ + beta p, S p = S r~ + beta S p_old, lambda += alpha p,
            // r -= alpha S p; the halo copies of p and r alike
            auto next_p = [&]() {
#pragma unroll
                for (int m = 0; m < R; ++m) {
                    s[m] = fma_rn(beta, t[m], q[m]);
                    p[m] = fma_rn(beta, p[m], z[m]);
                }
            };
            auto apply = [&]() {
#pragma unroll
                for (int m = 0; m < R; ++m) {
                    r[m] = fma_rn(-alpha, s[m], r[m]);
                    lam[m] = fma_rn(alpha, p[m], lam[m]);
                }
                if (st) {
                    put(vecR + own, r);
                    put(vecP + own, p);
                }
                // halo rows from one side (h: what it pushed), entry `base` of r and p
                auto halo_update = [&](const float *h, int base) {
                    float *vr = vecR + base, *vp = vecP + base;
                    for (int m = 0; m < R; ++m) {
                        vr[m] = fma_rn(-alpha, fma_rn(beta, h[halo_off(2, zpar, 0) + m], h[halo_off(1, zpar, 0) + m]), vr[m]);
                        vp[m] = fma_rn(beta, vp[m], h[halo_off(0, zpar, 0) + m]);
                    }
                };
                if (hany) {
                    if constexpr (PS) {
                        halo_update(hsrc, hbase);
                    } else {
#pragma unroll
                        for (int m = 0; m < R; ++m) {
                            hr[m] = fma_rn(-alpha, fma_rn(beta, ht[m], hq[m]), hr[m]);
                            hp[m] = fma_rn(beta, hp[m], hz[m]);
                        }
                        put(vecR + hbase, hr);
                        put(vecP + hbase, hp);
                    }
                }
                if (hboth) halo_update(halo + halo_off(0, 0, 1) + R * li, 2 * VSR + R * li);
            };
            if (!done) {
                next_p();
                if (!direct) apply();
            }
            recip.set(etan);
            g = beta;
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
                acc = exchange(dot(p, s), AT::zero(), AT::zero(), AT::zero()).eta;
                ups = AT::to_T(acc);
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
            for (int m = 0; m < R; ++m)
                if (R * li + m < NXR) P.lam[(size_t)(k0 + k) * NXR + R * li + m] = lam[m];
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

// The stages of one form; `after`: it may begin while the launch before it runs
static cudaError_t reg_stages(const PcgLaunch &L, PcgParams<float> P, bool after, cudaStream_t s) {
    P.kpc_max = L.kpc_max;
    P.n_upto = INT_MAX;
    cudaLaunchAttribute attr[2];
    PcgLaunch S = L;
    int full = 1;  // sizes of the stages: full, 3/4 full, 1/2 full
    while (full < L.C) full *= 2;
    const int mid = 3 * full / 4, low = full / 2;
    for (;; after = true) {
        const bool to_mid = P.queue && L.n_mid > 0 && S.C > mid, to_low = P.queue && L.n_mid > 0 && S.C == mid;
        P.n_above = to_mid ? mid * L.kpc_max : to_low ? low * L.kpc_max : INT_MIN;
        P.split = to_mid || to_low ? 0 : L.split;
        cudaLaunchConfig_t cfg = reg_config(S, S.clusters, attr, s);
        if (after) cfg.numAttrs = 2;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, reg_fn(S), P);
        if (e != cudaSuccess || !(to_mid || to_low)) return e;
        P.n_upto = P.n_above;
        P.queue += QUEUE_LEVELS;
        S.C = to_mid ? mid : low;
        S.clusters = to_mid ? L.n_mid : L.n_low;
    }
}

cudaError_t pcg_reg_launch(const PcgLaunch &L, const PcgParams<float> &P0, cudaStream_t s) {
    PcgParams<float> P = P0;
    const bool pick = L.light.clusters > 0 && P.queue;
    P.pick = pick ? 1 : 0;
    P.work = L.light.work;
    P.n_long = L.n_long;
    const cudaError_t e = reg_stages(L, P, false, s);
    if (e != cudaSuccess || !pick) return e;
    PcgLaunch R = L;
    R.reg = 1;
    R.C = L.light.C;
    R.clusters = L.light.clusters;
    R.n_mid = L.light.n_mid;
    R.n_low = L.light.n_low;
    R.split = L.light.split;
    R.kpc_max = L.light.kpc_max;
    R.threads = L.light.threads;
    R.smem = L.light.smem;
    P.pick = -1;
    return reg_stages(R, P, true, s);
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
