// Fine propagator of the FP32 mode on large grids (steady flow, n % 4 == 0): the method of
// fine_kernel.cuh in two passes and two group barriers a step instead of four, and 50 instead
// of 94 bytes a point (fused_kernel).
//
// The step starts from the previous increment, after which one BiCGStab iteration usually
// meets the tolerance (1.006 a step on the 64^3 Kolmogorov workload).  That first iteration
// has p = rhat = r, so with q = (A - I) r and q2 = (A - I) q
//     v = r + q,   s = (1 - alpha) r - alpha q,   (A - I) s = (1 - alpha) q - alpha q2,
// every dot product it needs follows from the six of r, q and q2, and its increment is
//     delta += alpha p + omega s.
// (The rounding of delta, r and the state is kept operation by operation as in fine_kernel: at
// 6e-8 of the increment it is what the FP32 mode's result is uncertain by.)
//   krylov : q and, from a ring of q planes in the same march, q2; only q is stored
//   setup  : of the next step: delta, u += delta and the residual r in one march
// The products are well scaled (1 - alpha is about ||q|| / ||r||); the scalars notice the few
// cases in which the sums cancel.  Where the residual is not predicted below the threshold, the
// step adds the increment, forms the true residual by another setup (without the state's
// update) and takes another iteration from there.
// The first step, whose start is far from its solution, is fine_kernel's (a launch of one step
// before this one; delta is u_1 - u_0), and so is the rest of an item from a step on that needs more
// than FUSED_MOST iterations (a launch after this one resumes it at the state before that step).
// The general iteration in this kernel would cost its registers (64^3 x 64, 40 steps: 12.1 ms with
// it, its spills reloaded in the marches, 7.6 without).
//
// What bounds it: latency and issue slots, not bytes (64^3 x 64: 4.4 TB/s of traffic, 41 % of
// the issue slots).  A CTA (one an SM, 256 threads with two units of four points each, so that
// two chains are in flight and the registers suffice) marches plane by plane with one CTA
// barrier a plane.  Inputs arrive as bulk copies of whole tile planes (rows of a tile are
// contiguous in memory; halo rows that wrap come as copies of their own), two or three planes
// ahead on mbarriers, so no registers hold loads in flight; six warps issue them, one array
// each, because one warp issuing all held the barrier up by 800 cycles a plane (8.2 -> 7.2 ms
// for 40 steps).  The state is kept as separate hi and lo planes and the arithmetic is packed in
// pairs (f32x2).  z neighbours stay in registers; the two halo rows of the operand are computed
// by a few warps, others each plane.
// Measured (GB300): the 64^3 Kolmogorov sweep, 64 x 157 steps, 58.4 -> 27.9 ms; 38 x 60
// steps of 128^3, 102 -> 42.5 ms; 96^3 x 16, 62 steps, 49.9 -> 13.2 ms.
#include "df.cuh"
#include "fine_kernel.cuh"

#include <algorithm>

namespace pr {

constexpr int FUSED_THREADS = 256;
constexpr int FU = 2;             // units of four points a thread works on in a tile plane
constexpr int FUSED_SSLOTS = 3;   // setup slots at most
constexpr int FUSED_RSLOTS = 6;   // planes of r in the krylov pass, three of them in use
// relative size below which a norm formed from products is not trusted (the products, summed in
// floats, hold ~1e-6)
constexpr double FUSED_CANCEL = 1e-4;
constexpr long long FUSED_DRAIN = 1 << 20;   // tries of a wait for copies in flight before leaving
// Iterations a step may take before its item is left to fine_kernel.  ms, fine_kernel alone and this
// kernel, by iterations a step: 64^3 x 64 x 40 steps 2.0 22.2 and 13.3, 3.0 30.7 and 19.4; x 16 6.6 and
// 4.5, 9.0 and 6.6; 96^3 x 16 x 40 2.0 41.5 and 14.0; 128^3 x 16 x 30 2.0 33.7 and 18.2.  From four on
// the iterations here, each restarted from the true residual, lose to fine_kernel's and the item goes
// back at its first such step, which then is done twice: x 30 steps 5.0 36.8 and 38.5, 8.7 59.9 and
// 62.1; limits of 5 and 9 only make that step longer (38.8, 39.4).
constexpr int FUSED_MOST = 3;

struct FusedShared : FineShared {
    float wred[5 * 32];
    float al, om, ga;   // alpha, omega, 1 - alpha of the last iteration: delta + al r + om (ga r - al q)
    int ok, its_max;
    int gave_up[2];     // a wait of an even, an odd plane gave up
    long long its_total;
    unsigned long long full[FUSED_SSLOTS + FUSED_RSLOTS];   // mbarriers: copies landed
};

// Four consecutive points as two packed pairs.
struct P4 { f2p a, b; };
__device__ __forceinline__ P4 ld4(const float* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ void st4(float* p, const P4& v) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.a, v.b); }
__device__ __forceinline__ P4 add4(const P4& x, const P4& y) { return {add2(x.a, y.a), add2(x.b, y.b)}; }
__device__ __forceinline__ P4 sub4(const P4& x, const P4& y) { return {sub2(x.a, y.a), sub2(x.b, y.b)}; }
__device__ __forceinline__ P4 mul4(const P4& x, const P4& y) { return {mul2(x.a, y.a), mul2(x.b, y.b)}; }
__device__ __forceinline__ P4 fma4(const P4& x, const P4& y, const P4& z) { return {fma2(x.a, y.a, z.a), fma2(x.b, y.b, z.b)}; }
__device__ __forceinline__ P4 fma4s(f2p x, const P4& y, const P4& z) { return {fma2(x, y.a, z.a), fma2(x, y.b, z.b)}; }
__device__ __forceinline__ P4 add4s(f2p x, const P4& y) { return {add2(x, y.a), add2(x, y.b)}; }
__device__ __forceinline__ P4 mul4s(f2p x, const P4& y) { return {mul2(x, y.a), mul2(x, y.b)}; }
__device__ __forceinline__ P4 pack4(const float (&v)[4]) { return {pk2(v[0], v[1]), pk2(v[2], v[3])}; }
__device__ __forceinline__ void unpack4(const P4& p, float (&v)[4]) {
    const float2 a = upk2(p.a), b = upk2(p.b);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ f2p both(float x) { return pk2(x, x); }
__device__ __forceinline__ P4 zero4() { return {0ull, 0ull}; }

// Arrival of a group's CTAs on a counter that only grows: one release and polls with acquire,
// no generation word (the reset and second word of group_barrier cost two more round trips to
// L2).  Thread 0 of each CTA calls it after a CTA barrier; `target` is the count that ends it.
__device__ __forceinline__ bool group_arrive_wait(unsigned* bar, unsigned target, long long spin_limit, int* err) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    for (long long i = 0;; ++i) {
        if ((int)(ld_acquire_u32(bar) - target) >= 0) return true;
        if (i >= spin_limit) {
            record_error(err, DERR_TIMEOUT);
            return false;
        }
        if (i >= 64) __nanosleep(64);
    }
}

// Sums over the group of NQ floats a thread (CTA by CTA in a fixed order), post(sums) in
// thread 0, all behind the group barrier number ep + 1.  Writes of the phase are visible to the
// group afterwards, also to its bulk copies (the proxy fences).
template <int NQ, typename Post>
__device__ __forceinline__ bool group_reduce(float (&v)[NQ], FusedShared& sh, double* part, int grid, int g0, int G,
                                             unsigned& ep, unsigned* bar, long long spin_limit, int* err, Post&& post) {
    constexpr int NV = NQ == 3 ? 4 : NQ;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float* red = sh.wred;
    asm volatile("fence.proxy.async;" ::: "memory");
    {
        float w[NV], s;
#pragma unroll
        for (int q = 0; q < NV; ++q) w[q] = q < NQ ? v[q < NQ ? q : 0] : 0.0f;
        const int q = chip_warp_sums(w, s);
        if (q >= 0) red[q * 32 + warp] = s;
    }
    __syncthreads();
    ++ep;
    double* mine = part + (size_t)(ep & 1) * 5 * grid;
    if (warp == 0) {
        double w[NV], s;
#pragma unroll
        for (int q = 0; q < NV; ++q) w[q] = lane < nw ? (double)red[q * 32 + lane] : 0.0;
        int q = chip_warp_sums(w, s);
        if (q >= 0 && q < NQ) mine[(size_t)q * grid + blockIdx.x] = s;
        __syncwarp();
        if (lane == 0) sh.ok = group_arrive_wait(bar, ep * (unsigned)G, spin_limit, err);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            w[k] = 0.0;
            if (k < NQ)
                for (int i = lane; i < G; i += 32) w[k] += __ldcg(mine + (size_t)k * grid + g0 + i);
        }
        q = chip_warp_sums(w, s);
        if (q >= 0) sh.sums[q] = s;
        __syncwarp();
        if (lane == 0) post(sh.sums);
        asm volatile("fence.proxy.async.global;" ::: "memory");
    }
    __syncthreads();
    return sh.ok != 0;
}

// One contiguous asynchronous copy, global to shared, counted on an mbarrier, and its
// bounded wait.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes), "r"((unsigned)__cvta_generic_to_shared(mbar))
                 : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* mbar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(mbar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned long long* mbar, unsigned parity, long long spin_limit) {
    const unsigned m = (unsigned)__cvta_generic_to_shared(mbar);
    for (long long i = 0; i <= spin_limit; ++i) {
        unsigned done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(m), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Shared memory: six float tables of n, the operand ring (three planes of TY + 2 rows:
// only the plane at the stencil is read, z neighbours being in registers), then the
// copies' slots: a setup slot holds TY + 2 rows of hi, lo, delta, r, q and TY of the forcing, a
// krylov slot TY + 4 rows of r.
struct FusedSmem {
    unsigned ring, slots, slot, total;   // bytes
};
__host__ __device__ inline FusedSmem fused_smem(int n, int TY, int slots) {
    FusedSmem f;
    f.ring = (6u * n * 4u + 127u) / 128u * 128u;
    f.slots = f.ring + 3u * (TY + 2) * n * 4u;
    f.slot = (5u * (TY + 2) + TY) * n * 4u;
    const unsigned s = slots * f.slot, k = FUSED_RSLOTS * (TY + 4) * n * 4u;
    f.total = f.slots + (s > k ? s : k);
    return f;
}

__global__ void __launch_bounds__(FUSED_THREADS, 1) fused_kernel(const __grid_constant__ FineArgs a) {
    extern __shared__ __align__(128) unsigned char smem_fused[];
    __shared__ FusedShared sh;
    const int G = a.G, g = blockIdx.x / G, q = blockIdx.x % G, grid = gridDim.x;
    const int n = a.g.n, n2 = n * n, TY = a.TY;
    const int lanes = n / 4, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int RT = (TY + FU - 1) / FU;   // this thread's rows: ty, ty + RT, ...
    const int ty = threadIdx.x / lanes;
    const int x0 = (threadIdx.x % lanes) * 4;
    const int xl = x0 == 0 ? n - 1 : x0 - 1, xr = x0 + 4 == n ? 0 : x0 + 4;
    const int TPN = a.NY * n;
    const int p_lo = (int)((long long)TPN * q / G), p_hi = (int)((long long)TPN * (q + 1) / G);
    const TileGeom geo{n, TY, p_lo, p_hi};
    const int t_lo = p_lo / n, t_hi = (p_hi + n - 1) / n;
    const int PL = (TY + 2) * n;             // floats of a ring plane
    bool act[FU];                            // owns a row of the tile there
    int so[FU];                              // its unit in a ring plane (0 if none)
#pragma unroll
    for (int u = 0; u < FU; ++u) {
        act[u] = ty < RT && ty + u * RT < TY;
        so[u] = act[u] ? (ty + u * RT + 1) * n + x0 : n + x0;
    }
    const FusedSmem fs = fused_smem(n, TY, a.fused_slots);
    float* tabk = reinterpret_cast<float*>(smem_fused);
    float* ring = reinterpret_cast<float*>(smem_fused + fs.ring);
    float* slots = reinterpret_cast<float*>(smem_fused + fs.slots);
    const unsigned Ng = (unsigned)a.g.Ng;
    // Krylov buffers of the group, by their offsets from Wk: delta and the residual in two
    // buffers each (a setup reads one at its neighbours while it writes the other), q; the rest
    // is the general iteration's
    float* Wk = reinterpret_cast<float*>(a.ws) + (size_t)g * FINE_NVEC * Ng;
    float* ust = reinterpret_cast<float*>(a.ust) + (size_t)g * 4 * Ng;   // two states: hi plane, lo plane
    unsigned xc = 0, xd = 7 * Ng, rc = Ng, rd = 2 * Ng;
    const unsigned qo = 5 * Ng;
    unsigned* bar = a.bar + 2 * (a.bar_groups + g);   // fine_kernel's barriers come first
    const int g0 = g * G;
    unsigned ep = 0;
    // the copies' slots in turn and the parity of their next landing
    const int NS = a.fused_slots;
    int ss = 0, rs = 0;
    unsigned sph = 0, rph = 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < FUSED_SSLOTS + FUSED_RSLOTS; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(&sh.full[i])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.gave_up[0] = sh.gave_up[1] = 0;
    }
    // What the launch after this one has to do for an item: nothing, until the item is done here.
    // Written before anything can wait: a wait that gives up then leaves no entry of an earlier
    // launch, or of uninitialised memory, behind.
    if (q == 0 && threadIdx.x == 0) {
        for (int b = g; b < a.B; b += a.numGroups) {
            int jb = 0, lb = b;
            while (jb + 1 < a.njobs && lb >= a.jobs[jb].B) lb -= a.jobs[jb++].B;
            a.jobs[jb].resume[lb] = 0;
        }
    }
    __syncthreads();
    // Waits for a slot's copies.  One that gives up says so in the entry of its plane's parity, which
    // is read after the plane's barrier and written again two barriers later, so that all threads
    // decide alike: they fill no slot again, wait for the copies in flight (`drain`: `count` slots of a
    // ring of `nring` from slot sl on, sl's landing of parity ph) and leave.  The group's other CTAs give
    // up at their next barrier.  (A vote at that barrier instead, __syncthreads_or, cost 4 %: 64^3 x 64 x 157 steps 27.9 -> 29.0 ms.)
    auto wait_full = [&](int i, unsigned parity, int plane) {
        if (!mbar_wait(&sh.full[i], parity, a.spin_limit)) {
            record_error(a.err, DERR_TIMEOUT);
            sh.gave_up[plane & 1] = 1;
        }
    };
    auto drain = [&](int first, int nring, int sl, unsigned ph, int count) {
        for (; count > 0; --count) {
            mbar_wait(&sh.full[first + sl], ph, FUSED_DRAIN);
            if (++sl == nring) {
                sl = 0;
                ph ^= 1;
            }
        }
    };
    auto wrapz = [&](int z) { return z < 0 ? z + n : (z >= n ? z - n : z); };
    // Rows y0 - hl .. y0 + TY + hl - 1 in at most three contiguous pieces: cnt rows from grid row
    // `row` to row `at` of the slot; piece 0 inside the grid, 1 and 2 wrapped below and above.
    auto piece_of = [&](int piece, int y0, int hl, int& row, int& cnt, int& at) {
        const int ya = max(y0 - hl, 0), yb = min(y0 + TY + hl, n);
        if (piece == 0) { row = ya; cnt = yb - ya; at = ya - (y0 - hl); }
        else if (piece == 1) { cnt = ya - (y0 - hl); row = n - cnt; at = 0; }
        else { cnt = y0 + TY + hl - yb; row = 0; at = TY + 2 * hl - cnt; }
    };
    // The 2 lanes halo units go to hw warps, beginning with warp hw0, which moves on each plane;
    // this thread's unit, or -1.
    const int hw = (2 * lanes + 31) >> 5;
    int hw0 = 0;
    auto halo_unit = [&]() {
        int w = warp - hw0;
        w = w < 0 ? w + nwarps : w;
        hw0 += hw;
        hw0 = hw0 >= nwarps ? hw0 - nwarps : hw0;
        const int u = w * 32 + lane;
        return u < 2 * lanes ? u : -1;
    };
    auto reduce = [&](auto& s, auto&& post) -> bool {
        return group_reduce<sizeof(s) / sizeof(float)>(s, sh, a.part, grid, g0, G, ep, bar, a.spin_limit, a.err, post);
    };

    int cur_job = -1;
    for (int b = g; b < a.B; b += a.numGroups) {
        int jb = 0, lb = b;
        while (jb + 1 < a.njobs && lb >= a.jobs[jb].B) lb -= a.jobs[jb++].B;
        const FineJob& J = a.jobs[jb];
        __syncthreads();
        if (jb != cur_job) {   // the velocity tables, scaled by dt / (2 h)
            cur_job = jb;
            for (int i = threadIdx.x; i < 6 * n; i += blockDim.x) tabk[i] = (float)(J.tab[i] * J.dt * 0.5 / a.g.h);
        }
        if (threadIdx.x == 0) {
            sh.status = 0;
            sh.its_total = 0;
            sh.its_max = 0;
        }
        __syncthreads();
        const float dtf = (float)J.dt, c1 = (float)(J.dt * J.eps / (a.g.h * a.g.h));
        const float* ff = J.f32;
        double* snap_b = J.snap ? reinterpret_cast<double*>(J.snap) + (size_t)lb * J.n_snap * Ng : nullptr;
        // the increment so far is delta + al r + om (ga r - al q)
        float al = 0.0f, om = 0.0f, ga = 0.0f;
        xc = 0, xd = 7 * Ng, rc = Ng, rd = 2 * Ng;
        int left = 0;                 // the step that is left to fine_kernel
        // owned points, a tile plane at a time
        auto owned = [&](auto&& fn) {
            for (int tt = t_lo; tt < t_hi; ++tt) {
                int y0, zlo, zhi;
                geo.tile(tt, y0, zlo, zhi);
#pragma unroll
                for (int u = 0; u < FU; ++u)
                    if (act[u])
                        for (int z = zlo; z < zhi; ++z) fn((unsigned)(z * n2 + (y0 - 1) * n + so[u]));
            }
        };
        if (J.S < 2 || J.status[lb] != 0) {   // no more steps, or fine_kernel's after a failed one
            if (q == 0 && threadIdx.x == 0) J.resume[lb] = J.S < 2 ? 0 : 2;
            continue;
        }
        // u_0 as a float pair, where the second step's setup reads its state, and the first step's
        // increment: u_1 is the pair u_0 + delta to 2^-48, so delta comes back to its last bit
        owned([&](unsigned i) {
            const Vec<double, 4> ud = vload<double, 4>(J.u_in + (size_t)lb * Ng + i);
            const Vec<double, 4> u1 = vload<double, 4>(J.u_out + (size_t)lb * Ng + i);
            float hi[4], lo[4], d[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 u = df_split(ud.v[e]);
                hi[e] = u.x;
                lo[e] = u.y;
                d[e] = (float)((u1.v[e] - (double)u.x) - (double)u.y);
            }
            st4(ust + i, pack4(hi));
            st4(ust + Ng + i, pack4(lo));
            st4(Wk + xc + i, pack4(d));
        });
        {
            float none[1] = {0.0f};
            if (!reduce(none, [](const double*) {})) return;
        }

        int j = 2, it = 0;
        while (j <= J.S) {
            const bool first = it == 0;   // of this step
            // ================ setup: delta, (first) u_{j-1} = u_{j-2} + delta, r = dt (f - L op) - delta
            // at op = u_{j-1} + delta
            {
                const unsigned uout = ((j - 1) & 1) * 2 * Ng, uin = first ? 2 * Ng - uout : uout;
                double* snap = (first && snap_b && (j - 1) % J.dM == 0 && (j - 1) / J.dM < J.n_snap)
                                   ? snap_b + (size_t)((j - 1) / J.dM) * Ng : nullptr;
                const bool upd = al != 0.0f;
                const f2p al2 = both(al), nal2 = both(-al), om2 = both(om), ga2 = both(ga), dt2 = both(dtf), c12 = both(c1);
                f2p f0 = 0ull, f1 = 0ull;   // sums of r^2 and (u + dt f)^2, the last planes' and all
                float s[2] = {0.0f, 0.0f};
                int ticks = 0;
                auto flush = [&]() {
                    const float2 x = upk2(f0), y = upk2(f1);
                    s[0] += x.x + x.y;
                    s[1] += y.x + y.y;
                    f0 = f1 = 0ull;
                    ticks = 0;
                };
                for (int tt = t_lo; tt < t_hi; ++tt) {
                    int y0, zlo, zhi;
                    geo.tile(tt, y0, zlo, zhi);
                    const int off = (y0 - 1) * n;   // + so[u]: in a plane of the grid
                    // negated velocity terms (row, x, and the sum along z)
                    float nxy[FU];
                    P4 nky, naz[FU];
                    {
                        float vy[4], vz[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) vy[e] = -tabk[TYX * n + x0 + e];
                        nky = pack4(vy);
#pragma unroll
                        for (int u = 0; u < FU; ++u) {
                            const int y = y0 + (act[u] ? ty + u * RT : 0);
                            nxy[u] = -tabk[TXY * n + y];
                            const float zy = tabk[TZY * n + y];
#pragma unroll
                            for (int e = 0; e < 4; ++e) vz[e] = -(tabk[TZX * n + x0 + e] + zy);
                            naz[u] = pack4(vz);
                        }
                    }
                    // Plane zp into a slot: warp w issues the pieces of array w (hi, lo, delta, r, q,
                    // forcing).  One warp issuing all of them would keep the others at the next
                    // barrier: the copies of a warp's lanes go out one after another.
                    auto issue = [&](int zp, int slot) {
                        float* sl = slots + slot * (fs.slot / 4);
                        unsigned long long* mb = &sh.full[slot];
                        const bool fin = ff && zp >= zlo && zp < zhi;
                        if (warp == 0 && lane == 0) {
                            const int planes = 3 + (upd ? 2 : 0);
                            mbar_expect(mb, (unsigned)((planes * PL + (fin ? TY * n : 0)) * 4));
                        }
                        for (int w = warp; w < 6; w += nwarps) {
                            if (w == 5) {
                                if (lane == 0 && fin) bulk_load(sl + 5 * PL, ff + zp * n2 + y0 * n, TY * n * 4, mb);
                            } else if (lane < 3 && (w < 3 || upd)) {
                                int row, cnt, at;
                                piece_of(lane, y0, 1, row, cnt, at);
                                const float* base = w < 2 ? ust + uin + w * Ng : Wk + (w == 2 ? xc : (w == 3 ? rc : qo));
                                if (cnt > 0) bulk_load(sl + w * PL + at * n, base + (wrapz(zp) * n2 + row * n), cnt * n * 4, mb);
                            }
                        }
                    };
                    // increment, state and operand of the unit at offset o of a slot
                    auto operand = [&](const float* sl, int o, P4& hi, P4& lo, P4& d) -> P4 {
                        hi = ld4(sl + o);
                        lo = ld4(sl + PL + o);
                        d = ld4(sl + 2 * PL + o);
                        if (upd) {
                            const P4 r = ld4(sl + 3 * PL + o);
                            const P4 sv = fma4s(nal2, ld4(sl + 4 * PL + o), mul4s(ga2, r));
                            d = fma4s(om2, sv, fma4s(al2, r, d));
                        }
                        if (first) {
                            // (hi, lo) + delta: TwoSum (Knuth) and the renormalising FastTwoSum
                            const P4 t = add4(hi, d), bb = sub4(t, hi);
                            const P4 e = add4(sub4(hi, sub4(t, bb)), sub4(d, bb));
                            const P4 l = add4(lo, e);
                            hi = add4(t, l);
                            lo = sub4(l, sub4(hi, t));
                        }
                        return add4(hi, add4(lo, d));
                    };
                    for (int d = 0, sl = ss; d < NS && zlo - 1 + d <= zhi; ++d) {
                        issue(zlo - 1 + d, sl);
                        sl = sl + 1 == NS ? 0 : sl + 1;
                    }
                    P4 um[FU], oc[FU], op[FU];   // operand at z - 1, z, z + 1
                    P4 dc[FU], fc[FU];           // delta and forcing at z
#pragma unroll
                    for (int u = 0; u < FU; ++u) oc[u] = op[u] = dc[u] = fc[u] = zero4();
                    float *rp = ring, *rq = ring + 2 * PL;   // ring planes of zp and of the stencil
                    for (int zp = zlo - 1; zp <= zhi; ++zp) {
                        wait_full(ss, sph, zp);
                        const float* sl = slots + ss * (fs.slot / 4);
                        const bool inside = zp >= zlo && zp < zhi;
                        P4 dn[FU], fn[FU];
#pragma unroll
                        for (int u = 0; u < FU; ++u) {
                            P4 hi, lo;
                            P4& d = dn[u];
                            um[u] = oc[u];
                            oc[u] = op[u];
                            op[u] = operand(sl, so[u], hi, lo, d);
                            fn[u] = zero4();
                            if (act[u]) {
                                st4(rp + so[u], op[u]);
                                if (inside) {
                                    const int i = zp * n2 + off + so[u];
                                    if (first) {
                                        st4(ust + uout + i, hi);
                                        st4(ust + uout + Ng + i, lo);
                                    }
                                    st4(Wk + xd + i, d);
                                    if (snap) {
                                        float hv[4], lv[4];
                                        unpack4(hi, hv);
                                        unpack4(lo, lv);
                                        Vec<double, 4> sd;
#pragma unroll
                                        for (int e = 0; e < 4; ++e) sd.v[e] = df_value_bits(hv[e], lv[e]);
                                        vstore(snap + i, sd);
                                    }
                                    if (ff) {
                                        fn[u] = ld4(sl + 5 * PL + so[u] - n);
                                        hi = fma4s(dt2, fn[u], hi);   // u + dt f
                                    }
                                    f1 = fma2(hi.a, hi.a, fma2(hi.b, hi.b, f1));
                                }
                            }
                        }
                        const int hu = halo_unit();
                        if (hu >= 0) {
                            const int o = hu < lanes ? hu * 4 : (TY + 1) * n + (hu - lanes) * 4;
                            P4 h_, l_, d_;
                            st4(rp + o, operand(sl, o, h_, l_, d_));
                        }
                        __syncthreads();
                        const int gave_up = sh.gave_up[zp & 1];
                        if (zp + NS <= zhi && !gave_up) issue(zp + NS, ss);
                        if (++ss == NS) {
                            ss = 0;
                            sph ^= 1;
                        }
                        if (zp > zlo) {
                            const int z = zp - 1;
                            const float nax = -tabk[TXZ * n + z], nay = -tabk[TYZ * n + z];
                            const P4 vy = add4s(both(nay), nky);
#pragma unroll
                            for (int u = 0; u < FU; ++u) {
                                if (!act[u]) continue;
                                const float* row = rq + so[u];
                                const P4 yp = ld4(row + n), ym = ld4(row - n);
                                const float el = row[xl - x0], er = row[xr - x0];
                                // differences to both sides (exact for close values), their sums and
                                // their differences: the x ones share the inner three
                                float c[4];
                                unpack4(oc[u], c);
                                const float d01 = __fsub_rn(c[1], c[0]), d12 = __fsub_rn(c[2], c[1]), d23 = __fsub_rn(c[3], c[2]);
                                const float dl = __fsub_rn(c[0], el), dr = __fsub_rn(er, c[3]);
                                const float gx[4] = {__fsub_rn(c[1], el), __fsub_rn(c[2], c[0]), __fsub_rn(c[3], c[1]),
                                                     __fsub_rn(er, c[2])};
                                const float lx[4] = {__fsub_rn(d01, dl), __fsub_rn(d12, d01), __fsub_rn(d23, d12),
                                                     __fsub_rn(dr, d23)};
                                const P4 gy = sub4(yp, ym), gz = sub4(op[u], um[u]);
                                const P4 ly = sub4(sub4(yp, oc[u]), sub4(oc[u], ym));
                                const P4 lz = sub4(sub4(op[u], oc[u]), sub4(oc[u], um[u]));
                                const P4 lap = add4(add4(pack4(lx), ly), lz);
                                P4 w = mul4s(both(nxy[u] + nax), pack4(gx));
                                w = fma4(naz[u], gz, fma4(vy, gy, w));
                                w = fma4s(c12, lap, fma4s(dt2, fc[u], w));
                                const P4 rv = sub4(w, dc[u]);
                                st4(Wk + rd + (z * n2 + off + so[u]), rv);
                                f0 = fma2(rv.a, rv.a, fma2(rv.b, rv.b, f0));
                            }
                            if (++ticks == 8) flush();
                        }
#pragma unroll
                        for (int u = 0; u < FU; ++u) {
                            dc[u] = dn[u];
                            fc[u] = fn[u];
                        }
                        rq = rp;
                        rp = rp == ring + 2 * PL ? ring : rp + PL;
                        if (gave_up) {   // planes zp .. zp + NS - 1 were on their way; ss is zp's next slot
                            const int sl = ss == 0 ? NS - 1 : ss - 1;
                            drain(0, NS, sl, ss == 0 ? sph ^ 1u : sph, min(NS, zhi - zp + 1));
                            return;
                        }
                    }
                    __syncthreads();   // the next tile rewrites the ring's first planes
                }
                flush();
                if (!reduce(s, [&](const double* d) {
                        const double rr0 = d[0], bb = d[1];
                        sh.thr = J.tol * sqrt(bb);
                        int conv = sqrt(rr0) <= sh.thr;
                        if (!isfinite(rr0) || !isfinite(bb)) {
                            sh.status = DERR_NONFINITE;
                            conv = 1;
                        }
                        sh.flag = conv;
                        sh.rho = rr0;
                    })) return;
                unsigned x = xc;
                xc = xd;
                xd = x;
                x = rc;
                rc = rd;
                rd = x;
            }
            al = om = ga = 0.0f;
            bool conv = sh.flag != 0;
            // ================ krylov: q = (A - I) r and the products of r, q, (A - I) q
            if (!conv) {
                const int RP_ = (TY + 4) * n;   // a plane of r; a unit's offset there: so + n
                const f2p c62 = both(6.0f * c1);
                f2p f[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
                float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
                int ticks = 0;
                auto flush = [&]() {
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        const float2 x = upk2(f[k]);
                        s[k] += x.x + x.y;
                        f[k] = 0ull;
                    }
                    ticks = 0;
                };
                for (int tt = t_lo; tt < t_hi; ++tt) {
                    int y0, zlo, zhi;
                    geo.tile(tt, y0, zlo, zhi);
                    const int off = (y0 - 1) * n;
                    // weights of the z neighbours, and what the y and x ones add to their plane's
                    float xy[FU];
                    P4 ky, wzp[FU], wzm[FU];
                    {
                        float vy[4], vp[4], vm[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) vy[e] = tabk[TYX * n + x0 + e];
                        ky = pack4(vy);
#pragma unroll
                        for (int u = 0; u < FU; ++u) {
                            const int y = y0 + (act[u] ? ty + u * RT : 0);
                            xy[u] = tabk[TXY * n + y];
                            const float zy = tabk[TZY * n + y];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float az = tabk[TZX * n + x0 + e] + zy;
                                vp[e] = az - c1;
                                vm[e] = -(az + c1);
                            }
                            wzp[u] = pack4(vp);
                            wzm[u] = pack4(vm);
                        }
                    }
                    auto issue = [&](int zp, int slot) {   // warp 0
                        float* sl = slots + slot * RP_;
                        unsigned long long* mb = &sh.full[FUSED_SSLOTS + slot];
                        if (lane == 0) mbar_expect(mb, (unsigned)(RP_ * 4));
                        __syncwarp();
                        if (lane < 3) {
                            int row, cnt, at;
                            piece_of(lane, y0, 2, row, cnt, at);
                            if (cnt > 0) bulk_load(sl + at * n, Wk + rc + wrapz(zp) * n2 + row * n, cnt * n * 4, mb);
                        }
                    };
                    // (A - I) at a unit: c its centre, e* the edges, ax, ay0 the plane's terms
                    auto opA = [&](const P4& c, float el, float er, const P4& yp, const P4& ym, const P4& zp, const P4& zm,
                                   float ax, float ay0, const P4& kyv, const P4& zpw, const P4& zmw) -> P4 {
                        float v[4];
                        unpack4(c, v);
                        const float wp = ax - c1, wm = ax + c1;
                        const float xs[4] = {wp * v[1] - wm * el, wp * v[2] - wm * v[0], wp * v[3] - wm * v[1],
                                             wp * er - wm * v[2]};
                        P4 o = fma4s(c62, c, pack4(xs));
                        o = fma4(add4s(both(ay0 - c1), kyv), yp, o);
                        const P4 wy = add4s(both(ay0 + c1), kyv);
                        o = sub4(o, mul4(wy, ym));
                        o = fma4(zpw, zp, o);
                        return fma4(zmw, zm, o);
                    };
                    // slots of planes z - 1, z, z + 1 in turn
                    auto next = [&](int sl) { return sl + 1 == FUSED_RSLOTS ? 0 : sl + 1; };
                    if (warp == 0) {
                        int sl = rs;
                        for (int d = 0; d < FUSED_RSLOTS && zlo - 2 + d <= zhi + 1; ++d) {
                            issue(zlo - 2 + d, sl);
                            sl = next(sl);
                        }
                    }
                    auto landed = [&](int z) {   // waits for the next plane, in plane z's turn; its slot
                        const int sl = rs;
                        wait_full(FUSED_SSLOTS + sl, rph, z);
                        if (++rs == FUSED_RSLOTS) {
                            rs = 0;
                            rph ^= 1;
                        }
                        return sl;
                    };
                    int sm = 0, sc = landed(zlo - 1), sp = landed(zlo - 1);
                    P4 rm[FU], rv[FU], rp[FU], qm[FU], qc[FU], qp[FU];   // r at z-1, z, z+1; q at z-2, z-1, z
#pragma unroll
                    for (int u = 0; u < FU; ++u) {
                        rv[u] = ld4(slots + sc * RP_ + n + so[u]);
                        rp[u] = ld4(slots + sp * RP_ + n + so[u]);
                        qc[u] = qp[u] = zero4();
                    }
                    float *qpl = ring, *qcl = ring + 2 * PL;   // ring planes of z and z - 1
                    float axm = 0.0f, aym = 0.0f;              // the velocity terms of the plane before
                    for (int z = zlo - 1; z <= zhi; ++z) {
                        sm = sc;
                        sc = sp;
                        sp = landed(z);
                        const int zw = wrapz(z);
                        const float ax = tabk[TXZ * n + zw], ay0 = tabk[TYZ * n + zw];
                        const float* cpl = slots + sc * RP_;
#pragma unroll
                        for (int u = 0; u < FU; ++u) {
                            rm[u] = rv[u];
                            rv[u] = rp[u];
                            qm[u] = qc[u];
                            qc[u] = qp[u];
                            rp[u] = ld4(slots + sp * RP_ + n + so[u]);
                            const float* row = cpl + n + so[u];
                            qp[u] = opA(rv[u], row[xl - x0], row[xr - x0], ld4(row + n), ld4(row - n), rp[u], rm[u], xy[u] + ax,
                                        ay0, ky, wzp[u], wzm[u]);
                            if (act[u]) {
                                st4(qpl + so[u], qp[u]);
                                if (z >= zlo && z < zhi) st4(Wk + qo + (z * n2 + off + so[u]), qp[u]);
                            }
                        }
                        const int hu = halo_unit();
                        if (hu >= 0) {
                            const bool low = hu < lanes;
                            const int hx = (low ? hu : hu - lanes) * 4;
                            int yy = low ? y0 - 1 : y0 + TY;
                            yy = yy < 0 ? yy + n : (yy >= n ? yy - n : yy);
                            const int ho = (low ? 1 : TY + 2) * n + hx;   // in a plane of r
                            const float* row = cpl + ho;
                            const float zy = tabk[TZY * n + yy];
                            float vy[4], vp[4], vm[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float az = tabk[TZX * n + hx + e] + zy;
                                vy[e] = tabk[TYX * n + hx + e];
                                vp[e] = az - c1;
                                vm[e] = -(az + c1);
                            }
                            st4(qpl + ho - n, opA(ld4(row), row[hx == 0 ? n - 1 : -1], row[hx + 4 == n ? 4 - n : 4], ld4(row + n),
                                                  ld4(row - n), ld4(slots + sp * RP_ + ho), ld4(slots + sm * RP_ + ho),
                                                  tabk[TXY * n + yy] + tabk[TXZ * n + zw], ay0, pack4(vy), pack4(vp), pack4(vm)));
                        }
                        __syncthreads();
                        const int gave_up = sh.gave_up[z & 1];
                        if (warp == 0 && z - 1 + FUSED_RSLOTS <= zhi + 1 && !gave_up) issue(z - 1 + FUSED_RSLOTS, sm);
                        if (z > zlo) {   // q2 at z - 1
#pragma unroll
                            for (int u = 0; u < FU; ++u) {
                                if (!act[u]) continue;
                                const float* row = qcl + so[u];
                                const P4 q2 = opA(qc[u], row[xl - x0], row[xr - x0], ld4(row + n), ld4(row - n), qp[u], qm[u],
                                                  xy[u] + axm, aym, ky, wzp[u], wzm[u]);
                                f[0] = fma2(rm[u].a, qc[u].a, fma2(rm[u].b, qc[u].b, f[0]));
                                f[1] = fma2(qc[u].a, qc[u].a, fma2(qc[u].b, qc[u].b, f[1]));
                                f[2] = fma2(rm[u].a, q2.a, fma2(rm[u].b, q2.b, f[2]));
                                f[3] = fma2(qc[u].a, q2.a, fma2(qc[u].b, q2.b, f[3]));
                                f[4] = fma2(q2.a, q2.a, fma2(q2.b, q2.b, f[4]));
                            }
                            if (++ticks == 8) flush();
                        }
                        axm = ax;
                        aym = ay0;
                        qcl = qpl;
                        qpl = qpl == ring + 2 * PL ? ring : qpl + PL;
                        if (gave_up) {   // planes z - 1 .. z + 4 were on their way, from slot sm on
                            drain(FUSED_SSLOTS, FUSED_RSLOTS, sm, sm < rs ? rph : rph ^ 1u, min(FUSED_RSLOTS, zhi + 3 - z));
                            return;
                        }
                    }
                    __syncthreads();
                }
                flush();
                // alpha, omega and the stopping tests of the first iteration from d = <r,q>, <q,q>,
                // <r,q2>, <q,q2>, <q2,q2>; sh.flag: 1 the step is done, 0 its true residual decides,
                // 2 fine_kernel has to take it
                if (!reduce(s, [&](const double* d) {
                        const double rr = sh.rho, thr2 = sh.thr * sh.thr;
                        const double rv = rr + d[0];
                        sh.flag = 2;
                        if (!(rv > 0.0) || !isfinite(rv)) return;
                        const double inv = 1.0 / rv, al_ = rr * inv, ga_ = d[0] * inv;   // alpha, 1 - alpha
                        const double a2 = al_ * al_, g2 = ga_ * ga_, ag = al_ * ga_;
                        const double ss2 = g2 * rr - 2.0 * ag * d[0] + a2 * d[1];       // <s, s>
                        const double scale = g2 * rr + a2 * d[1];
                        sh.al = (float)al_;   // delta += alpha r
                        sh.ga = (float)ga_;
                        sh.om = 0.0f;
                        sh.flag = fmax(ss2, FUSED_CANCEL * scale) <= thr2;
                        if (sh.flag || !(ss2 > FUSED_CANCEL * scale)) return;
                        const double su = g2 * d[0] - ag * d[2] - ag * d[1] + a2 * d[3];   // <s, (A - I) s>
                        const double uu = g2 * d[1] - 2.0 * ag * d[3] + a2 * d[4];
                        const double tt = ss2 + 2.0 * su + uu;
                        if (!(tt > 0.0) || !isfinite(tt)) {
                            sh.flag = 2;
                            return;
                        }
                        const double in = 1.0 / tt, om_ = (ss2 + su) * in, o1 = (su + uu) * in;   // omega, 1 - omega
                        const double w0 = o1 * o1 * ss2, w2 = om_ * om_ * uu;
                        const double rr1 = w0 - 2.0 * o1 * om_ * su + w2;                         // ||s - omega t||^2
                        sh.om = (float)om_;
                        sh.flag = fmax(rr1, FUSED_CANCEL * (w0 + w2)) <= thr2;
                    })) return;
                ++it;
                conv = sh.flag == 1;
                if (sh.flag == 2 || (!conv && it >= min(J.maxit, FUSED_MOST))) {
                    left = j;
                    --it;
                    break;
                }
                al = sh.al;
                om = sh.om;
                ga = sh.ga;
                if (!conv) continue;
            }
            if (threadIdx.x == 0) {
                sh.its_total += it;
                sh.its_max = max(sh.its_max, it);
            }
            // a non-finite state would only propagate: skip the remaining steps
            if (sh.status == DERR_NONFINITE) break;
            ++j;
            it = 0;
        }
        // ---------------- u_S = u_{S-1} + delta and its snapshot; or u_{j-1} of the step left over
        {
            const int S = J.S;
            const unsigned uo = ((left ? left - 1 : S - 1) & 1) * 2 * Ng;
            double* snap_S = (!left && snap_b && S % J.dM == 0 && S / J.dM < J.n_snap) ? snap_b + (size_t)(S / J.dM) * Ng : nullptr;
            owned([&](unsigned i) {
                float hi[4], lo[4], d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                unpack4(ld4(ust + uo + i), hi);
                unpack4(ld4(ust + uo + Ng + i), lo);
                if (!left) unpack4(ld4(Wk + xc + i), d);
                if (al != 0.0f && !left) {
                    float r4[4], q4[4];
                    unpack4(ld4(Wk + rc + i), r4);
                    unpack4(ld4(Wk + qo + i), q4);
#pragma unroll
                    for (int e = 0; e < 4; ++e) d[e] = fmaf(om, fmaf(-al, q4[e], ga * r4[e]), fmaf(al, r4[e], d[e]));
                }
                Vec<double, 4> u;
#pragma unroll
                for (int e = 0; e < 4; ++e) u.v[e] = df_value(df_add(make_float2(hi[e], lo[e]), d[e]));
                vstore(J.u_out + (size_t)lb * Ng + i, u);
                if (snap_S) vstore(snap_S + i, u);
            });
        }
        if (q == 0 && threadIdx.x == 0) {
            J.status[lb] = sh.status;
            J.its_total[lb] += (int)sh.its_total;
            J.its_max[lb] = max(J.its_max[lb], sh.its_max);
            J.resume[lb] = left;
        }
    }
}

// Rows a tile takes and the launch's threads and shared memory; false: the grid does not suit
// the kernel (n % 4, a tile of fewer than eight rows, or fewer than 96 threads).
static bool fused_geom(int n, int* TY, int* threads, int* slots, size_t* smem) {
    if (n % 4 != 0) return false;
    const int lanes = n / 4;
    *TY = 0;
    for (int ty = 1; ty <= n; ++ty)
        if (n % ty == 0 && (ty + FU - 1) / FU * lanes <= FUSED_THREADS) *TY = ty;
    if (*TY < 8 || (*TY + FU - 1) / FU * lanes < 96) return false;
    *threads = ((*TY + FU - 1) / FU * lanes + 31) / 32 * 32;
    for (*slots = FUSED_SSLOTS; *slots >= 2; --*slots) {
        const FusedSmem f = fused_smem(n, *TY, *slots);
        *smem = f.total;
        if (*smem <= 224 * 1024) return true;
    }
    return false;
}

bool fine_fused_takes(int n) {
    int TY, threads, slots;
    size_t smem;
    return fused_geom(n, &TY, &threads, &slots, &smem);
}

// Groups of G CTAs, one CTA an SM: the G of the least estimated time a step, which is so many
// turns of the groups over the B items times the barriers and reductions (12,000 cycles) and the
// planes of a CTA with the ones beyond its ends (2,700 each at 2048 points; 64^3 x 64, 40 steps:
// G = 1 14.0, 2 7.2, 4 8.0, 9 9.5, 19 12 ms).
static int fused_group(int planes, int B, int max_groups, int sms) {
    double best = 0.0;
    int G = 1;
    for (int c = 1; c <= std::min(sms, planes); ++c) {
        const int groups = std::min(std::min(B, max_groups), sms / c);
        const double t = (double)((B + groups - 1) / groups) * (12000.0 + 2700.0 * ((planes + c - 1) / c + 3));
        if (c == 1 || t < best) {
            best = t;
            G = c;
        }
    }
    return G;
}

void fine_fused_groups(int n, int B, int sms, std::vector<int>* out) {
    int TY, threads, slots;
    size_t smem;
    if (!fused_geom(n, &TY, &threads, &slots, &smem)) return;
    const int planes = n / TY * n, most = std::min(sms, planes);
    out->push_back(fused_group(planes, B, B, sms));
    out->push_back(std::max(1, std::min(sms / std::max(1, B), most)));   // all groups at once
    for (int c = 1; c <= most; c *= 2) out->push_back(c);
}

cudaError_t launch_fine_fused(FineArgs a, int max_groups, cudaStream_t st) {
    int threads;
    size_t smem;
    if (!fused_geom(a.g.n, &a.TY, &threads, &a.fused_slots, &smem)) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute((const void*)fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    a.RP = a.TY;
    a.NY = a.g.n / a.TY;
    const int planes = a.NY * a.g.n;
    int G = std::min(a.G, std::min(sms, planes));
    if (G <= 0) G = fused_group(planes, a.B, max_groups, sms);
    a.G = G;
    a.numGroups = std::min(std::min(a.B, max_groups), std::max(1, sms / G));
    void* args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void*)fused_kernel, dim3(G * a.numGroups), dim3(threads), args, smem, st);
    ++g_launch_count;
    return e;
}

}  // namespace pr
