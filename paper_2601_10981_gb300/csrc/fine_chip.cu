// Fine propagator on grids whose Krylov vectors fit the shared memory of one thread-block
// cluster (fine_chip_kernel).  The method, its stopping rule and its error codes are those
// of fine_kernel.cuh: implicit Euler in delta form, one BiCGStab solve per step.
//
// Measured (GB300): the 16^3 ABC workload's 125 FP64 steps of 8 subintervals 11.8 -> 3.7 ms.
// What bounds it: latency.  A 16^3 grid has 4096 points a subinterval; fine_kernel spends
// ~9.7 us a phase on it, almost all of it in its barrier through global memory (measured
// alone: 4500..6900 cycles), the reload of every vector from L2 at each phase, and the
// serial FP64 scalars.  GB300 issues one FP64 warp instruction per 64 cycles on each of an
// SM's four sub-partitions (dependent latency 64 cycles, a division 562, a square root 688),
// so in the FP64 mode the pipe is the second bound: every FP64 instruction counts, also the
// ones of a shuffle tree.
//
// Layout: a cluster of C CTAs owns one subinterval, CTA `rank` a slab of z-planes.  r, p, v
// and t stay in shared memory with one ghost plane on each side; delta, rhat, the state and
// the forcing (own points only) as well while they fit, otherwise in the global workspace
// (read and written once a step).  Operator weights come from per-row, per-plane and
// per-column tables in shared memory (FP64: 7 multiply-adds a point).
// A phase computes its vector at the owned points, stores the slab's first and last plane
// also into the neighbours' ghost planes (distributed shared memory) and its partial dot
// products into every CTA of the cluster, and ends at the hardware cluster barrier (365..500
// cycles).  Each CTA then sums the C partials in rank order, so all hold the same scalars.
// s = r - alpha v, r = s - omega t and p = r + beta (p - omega v) are recomputed on the ghost
// planes, so an iteration has two barriers: <rhat, v>, and the five products <t,s>, <t,t>,
// <s,s>, <rhat,s>, <rhat,t> that give omega and, by ||r||^2 = <s,s> - omega <t,s> and
// <rhat, r> = <rhat,s> - omega <rhat,t>, also the stopping test and beta (fine_kernel takes
// a third pass and barrier for those).
//
// No wait here polls memory: a cluster's CTAs are scheduled together and meet at the
// hardware barrier, which every thread reaches on every path (all branches depend on the
// shared scalars only).
#include "fine_kernel.cuh"

#include <algorithm>
#include <array>
#include <mutex>
#include <vector>

namespace pr {

constexpr int CHIP_MAXC = 16;
constexpr int CHIP_MAXWARPS = 16;
constexpr int CHIP_MAXQ = 5;
constexpr int CHIP_BATCH = 4;
constexpr size_t CHIP_SMEM = 224 * 1024;   // dynamic shared memory a CTA may use (beside ~2 KB static)

enum ChipKeep { CHIP_X = 1, CHIP_U = 2, CHIP_F = 4, CHIP_RH = 8 };   // held in shared memory

struct ChipPlan {
    int C, Cp;        // CTAs a cluster (<= n), the power of two not below
    int npl;          // planes of the largest slab, ceil(n / C)
    int keep;         // ChipKeep bits
    unsigned mpos, mlane;   // multipliers of the divisions by units-a-plane and units-a-row
};

template <typename KT>
struct ChipShared {
    KT red[CHIP_MAXQ * CHIP_MAXWARPS];
    double slot[2][CHIP_MAXQ][CHIP_MAXC];   // partials of all CTAs, alternating
    double tot[8];
    double rho, inv_rv, iom, thr, thr2;
    KT al, om, be;   // alpha, omega, beta for the vector updates (rounded once a CTA)
    int safe, act, status;
};

// Tests of doubles on the integer pipe: an FP64 compare would wait 64 cycles for its pipe.
__device__ __forceinline__ unsigned chip_exp(double x) { return ((unsigned)__double2hiint(x) >> 20) & 0x7ffu; }
__device__ __forceinline__ bool chip_finite(double x) { return chip_exp(x) != 0x7ffu; }
__device__ __forceinline__ bool chip_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
// a <= b for finite a and b >= 0
__device__ __forceinline__ bool chip_le(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }

// What follows a stopping test.
enum ChipAct { CHIP_GO = 0, CHIP_FULL = 1, CHIP_HALF = 2, CHIP_KEEP = 3, CHIP_CHECK = 4 };
// ||r||^2 = <s,s> - omega <t,s> below 2^-17 of <s,s> is not trusted in the FP32 mode, whose sums hold
// about 2^-20: unless even that would meet the threshold, r is formed and summed (CHIP_CHECK).  It
// happens where half a step cuts the residual several hundredfold, as on a first step from rest.
constexpr unsigned CHIP_CANCEL = 17;

__device__ __forceinline__ void chip_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned chip_cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Generic address of the same shared-memory object in CTA `rank` of the cluster.
template <typename T>
__device__ __forceinline__ T* chip_peer(T* p, unsigned rank) {
    unsigned long long o;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(o) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<T*>(o);
}

template <typename KT, int W, bool PT>
__global__ void __launch_bounds__(512, 1) fine_chip_kernel(FineArgs a, ChipPlan cp) {
    constexpr bool DF = std::is_same<KT, float>::value;   // double-float state
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ ChipShared<KT> sh;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int nw = nthr >> 5;
    const int n = a.g.n, n2 = n * n, C = cp.C;
    const long long Ng = a.g.Ng;
    const unsigned rank = chip_cluster_rank();
    const int cl = blockIdx.x / C;   // this cluster
    const int z0 = (int)((long long)n * rank / C), npl = (int)((long long)n * (rank + 1) / C) - z0;
    const unsigned below = (rank + C - 1) % C, above = (rank + 1) % C;
    const int lanes = n / W, npos = n * lanes;   // units (W points along x) of a row, of a plane

    // shared memory: r, p, t as [ghost below | ghost above | slab], v with two pairs of ghost
    // planes used in turn (a neighbour may still read the pair of the previous iteration)
    const int ar = (cp.npl + 2) * n2;
    KT* R = reinterpret_cast<KT*>(smem_raw);
    KT* P = R + ar;
    KT* T = P + ar;
    KT* V = T + ar;
    KT* next = V + ar + 2 * n2;
    const int own = 2 * n2;   // offset of the slab
    KT* X = nullptr;
    KT* RH = nullptr;
    KT* Fs = nullptr;
    using ST = typename std::conditional<DF, float2, double>::type;
    ST* U = nullptr;
    if (cp.keep & CHIP_U) {
        U = reinterpret_cast<ST*>(next);
        next = reinterpret_cast<KT*>(U + cp.npl * n2);
    }
    if (cp.keep & CHIP_X) { X = next; next += cp.npl * n2; }
    if (cp.keep & CHIP_F) { Fs = next; next += cp.npl * n2; }
    if (cp.keep & CHIP_RH) { RH = next; next += cp.npl * n2; }
    // operator tables.  FP64: the weights of the six neighbours; FP32: dt b_d / (2h)
    KT* ax = next;                          // [slab plane][y]
    KT* ay = ax + cp.npl * n;               // [slab plane][x]
    KT* az = ay + cp.npl * n;               // [y][x]
    KT* bx = az + n2;                       // FP64: the weights at the lower neighbours
    KT* by = bx + cp.npl * n;
    KT* bz = by + cp.npl * n;
    // own-point vectors that did not fit: this cluster's part of the global workspace
    if (!X) X = reinterpret_cast<KT*>(a.ws) + (size_t)cl * FINE_NVEC * Ng + (size_t)z0 * n2;
    if (!RH) RH = reinterpret_cast<KT*>(a.ws) + ((size_t)cl * FINE_NVEC + 2) * Ng + (size_t)z0 * n2;
    if (!U) U = reinterpret_cast<ST*>(a.ust + (size_t)cl * 2 * Ng) + (size_t)z0 * n2;
    KT* const Rb = chip_peer(R, below) + n2;      // my first plane is their ghost above
    KT* const Ra = chip_peer(R, above);           // my last plane is their ghost below
    KT* const Tb = chip_peer(T, below) + n2;
    KT* const Ta = chip_peer(T, above);
    KT* const Vb = chip_peer(V, below) + n2;
    KT* const Va = chip_peer(V, above);

    const double h = a.g.h;
    int par = 0;      // which half of sh.slot the next reduction fills
    int vg = 0;       // which pair of ghost planes of v is current
    double dt = 0.0;
    KT c1 = (KT)0, c0 = (KT)1;
    const KT* bpk = nullptr;   // stored velocity perturbation
    KT kp = (KT)0;
    int cur_job = -1;
    (void)bpk;
    (void)kp;

    auto push = [&](KT* lo, KT* hi, int o, const Vec<KT, W>& v) {   // o: index within the slab
        if (o < n2) vstore(lo + o, v);
        if (o >= (npl - 1) * n2) vstore(hi + (o - (npl - 1) * n2), v);
    };
    // v at flat index i of [ghost below | ghost above | slab]
    auto vptr = [&](int i) -> KT* { return V + (i < own ? vg * own + i : own + i); };

    // Sums over the cluster of NQ values a thread, then post(totals) on warp 0.  Ends with
    // every thread past a CTA barrier; ghost planes pushed before the call are visible.
    auto reduce = [&](auto& acc, auto&& post) {
        constexpr int NQ = sizeof(acc) / sizeof(acc[0]);
        {
            KT s;
            const int q = chip_warp_sums(acc, s);
            if (q >= 0) sh.red[q * CHIP_MAXWARPS + warp] = s;
        }
        __syncthreads();
        {
            int nwp = 1;
            while (nwp < nw) nwp *= 2;
            const int per = 32 / nwp;
            const int q = warp * per + lane / nwp, w = lane % nwp;
            if (warp * per < NQ) {
                double x = (q < NQ && w < nw) ? (double)sh.red[q * CHIP_MAXWARPS + w] : 0.0;
                for (int o = nwp / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (q < NQ)
                    for (int c = w; c < C; c += nwp) *chip_peer(&sh.slot[par][q][rank], c) = x;
            }
        }
        chip_cluster_sync();
        const int Cp = cp.Cp, per = 32 / Cp;
        if (warp * per < NQ) {
            const int q = warp * per + lane / Cp, c = lane % Cp;
            double x = (q < NQ && c < C) ? sh.slot[par][q][c] : 0.0;
            for (int o = Cp / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (q < NQ && c == 0) sh.tot[q] = x;
        }
        if (NQ * Cp > 32) __syncthreads();
        else __syncwarp();
        if (warp == 0) post();
        __syncthreads();
        par ^= 1;
    };
    // ||r||^2 = rr against the stopping threshold; by squares unless they could leave the range
    // (rr finite)
    auto met = [&](double rr) -> bool {
        return sh.safe ? chip_le(rr, sh.thr2) : sqrt(fmax(rr, 0.0)) <= sh.thr;
    };

    // stencils: fn(o, ip, zl, y, x0, nb) for each owned unit, o its index within the slab
    auto stencil = [&](const KT* A, auto&& fn) {
        for (int u = tid; u < npl * npos; u += nthr) {
            const int z = (int)__umulhi((unsigned)u, cp.mpos);
            const int ps = u - z * npos;
            const int y = lanes == 1 ? ps : (int)__umulhi((unsigned)ps, cp.mlane);
            const int x0 = (ps - y * lanes) * W;
            const KT* S = A + own + z * n2;
            const KT* row = S + y * n;
            Nb7<KT, W> q;
            q.c = vload<KT, W>(row + x0);
#pragma unroll
            for (int e = 0; e < W - 1; ++e) {
                q.xp.v[e] = q.c.v[e + 1];
                q.xm.v[e + 1] = q.c.v[e];
            }
            q.xp.v[W - 1] = row[x0 + W == n ? 0 : x0 + W];
            q.xm.v[0] = row[x0 == 0 ? n - 1 : x0 - 1];
            q.yp = vload<KT, W>((y + 1 == n ? S : row + n) + x0);
            q.ym = vload<KT, W>((y == 0 ? S + n2 - n : row - n) + x0);
            q.zp = vload<KT, W>((z + 1 == npl ? A + n2 : S + n2) + y * n + x0);
            q.zm = vload<KT, W>((z == 0 ? A : S - n2) + y * n + x0);
            fn(z * n2 + y * n + x0, z, y, x0, q);
        }
    };
    // The neighbours' weights of A = I + dt L at point e of a unit: up[d], dn[d].
    auto weights = [&](int o, int z, int y, int x, KT (&up)[3], KT (&dn)[3]) {
        if constexpr (DF) {
            const KT w[3] = {ax[z * n + y], ay[z * n + x], az[y * n + x]};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                KT t = w[d];
                if constexpr (PT) t += kp * bpk[(size_t)d * Ng + (size_t)z0 * n2 + o];
                up[d] = t - c1;
                dn[d] = -(t + c1);
            }
        } else {
            up[0] = ax[z * n + y], up[1] = ay[z * n + x], up[2] = az[y * n + x];
            dn[0] = bx[z * n + y], dn[1] = by[z * n + x], dn[2] = bz[y * n + x];
            if constexpr (PT) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const KT t = kp * bpk[(size_t)d * Ng + (size_t)z0 * n2 + o];
                    up[d] += t;
                    dn[d] -= t;
                }
            }
        }
    };
    auto applyA = [&](int o, int z, int y, int x0, const Nb7<KT, W>& q) -> Vec<KT, W> {
        Vec<KT, W> r;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            KT up[3], dn[3];
            weights(o + e, z, y, x0 + e, up, dn);
            r.v[e] = c0 * q.c.v[e] + up[0] * q.xp.v[e] + dn[0] * q.xm.v[e] + up[1] * q.yp.v[e] + dn[1] * q.ym.v[e] +
                     up[2] * q.zp.v[e] + dn[2] * q.zm.v[e];
        }
        return r;
    };

    chip_cluster_sync();   // every CTA of the cluster runs: its shared memory may be written
    // The products of the second half of an iteration, <rhat, s> with NQ = 5 (FINE_EARLY)
    auto dots2 = [](auto& s, KT tv, KT sv, KT hv) {
        s[0] += tv * sv;
        s[1] += tv * tv;
        s[2] += sv * sv;
        s[3] += hv * tv;
        if constexpr (sizeof(s) / sizeof(s[0]) == 5) s[4] += hv * sv;
    };
    for (int b = cl; b < a.B; b += gridDim.x / C) {
        int jb = 0, lb = b;
        while (jb + 1 < a.njobs && lb >= a.jobs[jb].B) lb -= a.jobs[jb++].B;
        const FineJob& J = a.jobs[jb];
        if (jb != cur_job) {
            // no stencil of the previous item is running: all are past a cluster barrier
            cur_job = jb;
            dt = J.dt;
            const double sc = J.dt * 0.5 / h, d1 = J.dt * J.eps / (h * h);
            c1 = (KT)d1;
            c0 = (KT)(1.0 + 6.0 * dt * J.eps / (h * h));
            if constexpr (PT) {
                bpk = reinterpret_cast<const KT*>(J.pert);
                kp = (KT)sc;
            }
            const double* tb = J.tab;
            // velocity va + vb.  FP32: each part scaled and rounded by itself, as fine_kernel does
            auto put = [&](KT* up, KT* dn, int i, double va, double vb) {
                if constexpr (DF) {
                    up[i] = (KT)(va * J.dt * 0.5 / h) + (KT)(vb * J.dt * 0.5 / h);
                } else {
                    up[i] = (va + vb) * sc - d1;
                    dn[i] = -((va + vb) * sc + d1);
                }
            };
            for (int i = tid; i < npl * n; i += nthr) {
                const int z = i / n, k = i - z * n;
                put(ax, bx, i, tb[TXY * n + k], tb[TXZ * n + z0 + z]);
                put(ay, by, i, tb[TYX * n + k], tb[TYZ * n + z0 + z]);
            }
            for (int i = tid; i < n2; i += nthr) {
                const int y = i / n, x = i - y * n;
                put(az, bz, i, tb[TZX * n + x], tb[TZY * n + y]);
            }
        }
        const int S = J.S, dM = J.dM, n_snap = J.n_snap;
        const double tol2 = J.tol * J.tol;
        const KT dtk = (KT)dt;
        const size_t slab = (size_t)lb * Ng + (size_t)z0 * n2;
        double* snap_b = J.snap ? reinterpret_cast<double*>(J.snap) + (size_t)lb * n_snap * Ng + (size_t)z0 * n2 : nullptr;
        double* outp = J.u_out + slab;
        const KT* fg;
        if constexpr (DF) fg = J.f32;
        else fg = J.f;
        const KT* F = fg ? fg + (size_t)z0 * n2 : nullptr;
        if (tid == 0) sh.status = 0;
        // u_0, its snapshot, and the operand of the first residual
        for (int o = tid * W; o < npl * n2; o += nthr * W) {
            const Vec<double, W> ud = vload<double, W>(J.u_in + slab + o);
            Vec<KT, W> op;
            Vec<ST, W> us;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                if constexpr (DF) {
                    us.v[e] = df_split(ud.v[e]);
                    op.v[e] = us.v[e].x;
                } else {
                    us.v[e] = ud.v[e];
                    op.v[e] = ud.v[e];
                }
            }
            vstore(U + o, us);
            vstore(T + own + o, op);
            push(Tb, Ta, o, op);
            if (snap_b && n_snap > 0) {
                Vec<double, W> sd;
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    if constexpr (DF) sd.v[e] = df_value_bits(us.v[e].x, us.v[e].y);
                    else sd.v[e] = us.v[e];
                }
                vstore(snap_b + o, sd);
            }
            if (Fs && F) vstore(Fs + o, vload<KT, W>(F + o));
        }
        const KT* Fp = F ? (Fs ? Fs : F) : nullptr;
        long long its_total = 0;
        int its_max = 0;
        bool dvalid = false;

        for (int j = 1; j <= S; ++j) {
            // ---- residual of u_{j-1}; the FP32 mode starts from the previous increment
            const bool xg = DF && dvalid;
            chip_cluster_sync();   // the operand's ghost planes are in place
            {
                KT acc[2] = {(KT)0, (KT)0};
                stencil(T, [&](int o, int z, int y, int x0, const Nb7<KT, W>& q) {
                    Vec<KT, W> fv, rv;
                    if (Fp) fv = vload<KT, W>(Fp + o);
                    else {
#pragma unroll
                        for (int e = 0; e < W; ++e) fv.v[e] = (KT)0;
                    }
                    if constexpr (DF) {
                        Vec<KT, W> dv;
                        if (xg) dv = vload<KT, W>(X + o);
                        else {
#pragma unroll
                            for (int e = 0; e < W; ++e) dv.v[e] = (KT)0;
                        }
                        const Vec<float2, W> us = vload<float2, W>(reinterpret_cast<const float2*>(U) + o);
                        KT s0 = (KT)0, s1 = (KT)0;
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            const float c = q.c.v[e];
                            KT w0 = ax[z * n + y], w1 = ay[z * n + x0 + e], w2 = az[y * n + x0 + e];
                            if constexpr (PT) {
                                const size_t g = (size_t)z0 * n2 + o + e;
                                w0 += kp * bpk[g];
                                w1 += kp * bpk[Ng + g];
                                w2 += kp * bpk[2 * Ng + g];
                            }
                            const KT dx = __fsub_rn(q.xp.v[e], q.xm.v[e]);
                            const KT dy = __fsub_rn(q.yp.v[e], q.ym.v[e]);
                            const KT dz = __fsub_rn(q.zp.v[e], q.zm.v[e]);
                            const KT sx = __fsub_rn(__fsub_rn(q.xp.v[e], c), __fsub_rn(c, q.xm.v[e]));
                            const KT sy = __fsub_rn(__fsub_rn(q.yp.v[e], c), __fsub_rn(c, q.ym.v[e]));
                            const KT sz = __fsub_rn(__fsub_rn(q.zp.v[e], c), __fsub_rn(c, q.zm.v[e]));
                            const KT rk =
                                (dtk * fv.v[e] - (w0 * dx + w1 * dy + w2 * dz) + c1 * ((sx + sy) + sz)) - dv.v[e];
                            rv.v[e] = rk;
                            const KT bi = us.v[e].x + dtk * fv.v[e];
                            s0 += rk * rk;
                            s1 += bi * bi;
                        }
                        acc[0] += s0;
                        acc[1] += s1;
                    } else {
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            // dt L u from differences to the centre (the weights of L add up
                            // to zero), so rounding scales with the differences
                            KT up[3], dn[3];
                            weights(o + e, z, y, x0 + e, up, dn);
                            const KT c = q.c.v[e];
                            const KT Lu = up[0] * (q.xp.v[e] - c) + dn[0] * (q.xm.v[e] - c) + up[1] * (q.yp.v[e] - c) +
                                          dn[1] * (q.ym.v[e] - c) + up[2] * (q.zp.v[e] - c) + dn[2] * (q.zm.v[e] - c);
                            const KT rk = Fp ? dtk * fv.v[e] - Lu : -Lu;
                            rv.v[e] = rk;
                            const KT bi = Fp ? c + dtk * fv.v[e] : c;
                            acc[0] += rk * rk;
                            acc[1] += bi * bi;
                        }
                    }
                    vstore(R + own + o, rv);
                    push(Rb, Ra, o, rv);
                });
                reduce(acc, [&]() {
                    if (lane == 0) {
                        const double rr0 = sh.tot[0], bb = sh.tot[1];
                        const bool safe = chip_exp(bb) > 360u && chip_exp(bb) < 1686u;   // 2^-663 .. 2^663
                        sh.safe = safe;
                        sh.thr2 = tol2 * bb;
                        if (!safe) sh.thr = J.tol * sqrt(bb);
                        int act = CHIP_GO;
                        if (!chip_finite(rr0) || !chip_finite(bb)) {
                            sh.status = DERR_NONFINITE;
                            act = CHIP_KEEP;
                        } else if (met(rr0)) {
                            act = CHIP_KEEP;
                        }
                        sh.rho = rr0;
                        sh.act = act;
                    }
                });
            }
            int it = 0;
            int act = sh.act;
            while (act == CHIP_GO) {
                ++it;
                const bool first = it == 1;
                vg ^= 1;
                // ---- v = A p (first iteration: p = r = rhat)
                {
                    KT acc[1] = {(KT)0};
                    stencil(first ? R : P, [&](int o, int z, int y, int x0, const Nb7<KT, W>& q) {
                        const Vec<KT, W> av = applyA(o, z, y, x0, q);
                        vstore(V + 2 * own + o, av);
                        push(Vb + vg * own, Va + vg * own, o, av);
                        Vec<KT, W> hv = q.c;
                        if (!first) hv = vload<KT, W>(RH + o);
                        if constexpr (W == 1) {
                            acc[0] += hv.v[0] * av.v[0];
                        } else {
                            KT s = (KT)0;
#pragma unroll
                            for (int e = 0; e < W; ++e) s += hv.v[e] * av.v[e];
                            acc[0] += s;
                        }
                    });
                    reduce(acc, [&]() {
                        const double rv = sh.tot[0];
                        const double qv = (lane == 0 ? sh.rho : 1.0) / rv;
                        if (lane == 1) sh.inv_rv = qv;
                        if (lane == 0) {
                            if (chip_zero(rv) || !chip_finite(rv)) {
                                sh.status = chip_finite(rv) ? DERR_BREAKDOWN : DERR_NONFINITE;
                                sh.act = CHIP_KEEP;
                            } else {
                                sh.al = (KT)qv;
                                sh.act = CHIP_GO;
                            }
                        }
                    });
                }
                if (sh.act != CHIP_GO) {
                    --it;
                    break;
                }
                // ---- s = r - alpha v (ghost planes too), t = A s
                {
                    const KT al = sh.al;
                    // (loads of CHIP_BATCH units first: a store would hold back the loads behind it)
                    const int end = own + npl * n2;
                    for (int i0 = tid * W; i0 < end; i0 += CHIP_BATCH * nthr * W) {
                        Vec<KT, W> rv[CHIP_BATCH], vv[CHIP_BATCH];
#pragma unroll
                        for (int k = 0; k < CHIP_BATCH; ++k) {
                            const int i = i0 + k * nthr * W;
                            if (i < end) {
                                rv[k] = vload<KT, W>(R + i);
                                vv[k] = vload<KT, W>(vptr(i));
                            }
                        }
#pragma unroll
                        for (int k = 0; k < CHIP_BATCH; ++k) {
                            const int i = i0 + k * nthr * W;
                            if (i >= end) break;
                            if (first) vstore(P + i, rv[k]);
#pragma unroll
                            for (int e = 0; e < W; ++e) rv[k].v[e] -= al * vv[k].v[e];
                            vstore(R + i, rv[k]);
                        }
                    }
                    __syncthreads();
                    // what follows from ||r||^2 and <rhat, r>; beta and rho if another iteration does
                    auto after = [&](double rr1, double rho_new, double iom) -> int {
                        if (!chip_finite(rr1)) {
                            sh.status = DERR_NONFINITE;
                        } else if (met(rr1)) {
                        } else if (chip_zero(rho_new)) {
                            sh.status = DERR_BREAKDOWN;
                        } else if (it >= J.maxit) {
                            sh.status = DERR_NOT_CONVERGED;
                        } else {
                            sh.be = (KT)(rho_new * iom * sh.inv_rv);   // (rho'/rho)(alpha/omega)
                            sh.rho = rho_new;
                            return CHIP_GO;
                        }
                        return CHIP_FULL;
                    };
                    auto half = [&](auto& acc) {
                        constexpr int NQ = sizeof(acc) / sizeof(acc[0]);
                        stencil(R, [&](int o, int z, int y, int x0, const Nb7<KT, W>& q) {
                            const Vec<KT, W> tv = applyA(o, z, y, x0, q);
                            vstore(T + own + o, tv);
                            push(Tb, Ta, o, tv);
                            const Vec<KT, W> hv = vload<KT, W>(first ? P + own + o : RH + o);
                            [[maybe_unused]] KT s[NQ] = {};
    #pragma unroll
                            for (int e = 0; e < W; ++e) {
                                if constexpr (W == 1) {
                                    dots2(acc, tv.v[e], q.c.v[e], hv.v[e]);
                                } else {
                                    dots2(s, tv.v[e], q.c.v[e], hv.v[e]);
                                }
                            }
                            if constexpr (W > 1) {
    #pragma unroll
                                for (int k = 0; k < NQ; ++k) acc[k] += s[k];
                            }
                        });
                        reduce(acc, [&]() {
                            const double ts = sh.tot[0], tt = sh.tot[1], ss = sh.tot[2];
                            const double qv = (lane == 0 ? ts : tt) / (lane == 0 ? tt : ts);   // omega, 1 / omega
                            const double iom = __shfl_sync(0xffffffffu, qv, 1);
                            if (lane == 0) {
                                int act2 = CHIP_GO;
                                double om = 0.0;
                                if (chip_finite(ss) && met(ss)) {
                                    act2 = CHIP_HALF;
                                } else if (chip_zero(tt) || !chip_finite(tt)) {
                                    sh.status = chip_finite(tt) ? DERR_BREAKDOWN : DERR_NONFINITE;
                                    act2 = CHIP_HALF;
                                } else {
                                    om = qv;
                                    if (chip_zero(om)) sh.status = DERR_BREAKDOWN;
                                    if (sh.status != 0) {
                                        act2 = CHIP_HALF;
                                    } else {
                                        const double rr1 = fma(-om, ts, ss);                    // ||s - omega t||^2
                                        const double rho_new = fma(-om, sh.tot[3], NQ == 5 ? sh.tot[4] : 0.0);   // <rhat, r>
                                        if (DF && chip_finite(rr1) && chip_exp(rr1) + CHIP_CANCEL < chip_exp(ss)) {
                                            act2 = met(0x1p-17 * ss) ? CHIP_FULL : CHIP_CHECK;
                                            sh.iom = iom;
                                        } else {
                                            act2 = after(rr1, rho_new, iom);
                                        }
                                    }
                                }
                                sh.om = (KT)om;
                                sh.act = act2;
                            }
                        });
                    };
                    if (DF || it > FINE_EARLY) {
                        KT acc[5] = {};
                        half(acc);
                    } else {
                        KT acc[4] = {};
                        half(acc);
                    }
                    if (DF && sh.act == CHIP_CHECK) {
                        const KT om = sh.om;
                        KT chk[2] = {(KT)0, (KT)0};
                        for (int o = tid * W; o < npl * n2; o += nthr * W) {
                            const Vec<KT, W> sv = vload<KT, W>(R + own + o), tv = vload<KT, W>(T + own + o);
                            const Vec<KT, W> hv = vload<KT, W>(first ? P + own + o : RH + o);
#pragma unroll
                            for (int e = 0; e < W; ++e) {
                                const KT rn = sv.v[e] - om * tv.v[e];
                                chk[0] += rn * rn;
                                chk[1] += hv.v[e] * rn;
                            }
                        }
                        reduce(chk, [&]() {
                            if (lane == 0) sh.act = after(sh.tot[0], sh.tot[1], sh.iom);
                        });
                    }
                }
                act = sh.act;
                if (act != CHIP_GO) break;
                // ---- delta += alpha p + omega s, r = s - omega t, p = r + beta (p - omega v)
                {
                    const KT al = sh.al, om = sh.om, be = sh.be;
                    const bool x0z = first && !xg;   // delta starts from zero
                    for (int i = tid * W; i < own + npl * n2; i += nthr * W) {
                        const Vec<KT, W> s = vload<KT, W>(R + i), t = vload<KT, W>(T + i), p = vload<KT, W>(P + i);
                        const Vec<KT, W> v = vload<KT, W>(vptr(i));
                        Vec<KT, W> rn, pn;
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            rn.v[e] = s.v[e] - om * t.v[e];
                            pn.v[e] = rn.v[e] + be * (p.v[e] - om * v.v[e]);
                        }
                        vstore(R + i, rn);
                        vstore(P + i, pn);
                        if (i >= own) {
                            const int o = i - own;
                            Vec<KT, W> x;
                            if (!x0z) x = vload<KT, W>(X + o);
#pragma unroll
                            for (int e = 0; e < W; ++e) x.v[e] = (x0z ? (KT)0 : x.v[e]) + al * p.v[e] + om * s.v[e];
                            vstore(X + o, x);
                            if (first) vstore(RH + o, p);
                        }
                    }
                    __syncthreads();
                }
            }
            // `act` of a break at <rhat, v> stays CHIP_GO above: nothing is added to delta
            const int fin = (act == CHIP_FULL || act == CHIP_HALF) ? act : CHIP_KEEP;
            dvalid = it > 0 || xg;
            its_total += it;
            its_max = max(its_max, it);
            const int status = sh.status;
            // ---- u_j = u_{j-1} + delta, its snapshot or output, and the next operand
            {
                const KT al = sh.al, om = sh.om;
                const bool x0z = it <= 1 && !xg;   // delta holds nothing yet
                const bool last = j == S || status == DERR_NONFINITE;
                double* snap_j = (snap_b && j % dM == 0 && j / dM < n_snap) ? snap_b + (size_t)(j / dM) * Ng : nullptr;
                for (int o = tid * W; o < npl * n2; o += nthr * W) {
                    Vec<KT, W> x;
                    if (!dvalid || (x0z && fin != CHIP_KEEP)) {
#pragma unroll
                        for (int e = 0; e < W; ++e) x.v[e] = (KT)0;
                    } else {
                        x = vload<KT, W>(X + o);
                    }
                    if (fin != CHIP_KEEP) {
                        const Vec<KT, W> p = vload<KT, W>(P + own + o);
                        if (fin == CHIP_FULL) {
                            const Vec<KT, W> s = vload<KT, W>(R + own + o);
#pragma unroll
                            for (int e = 0; e < W; ++e) x.v[e] = x.v[e] + al * p.v[e] + om * s.v[e];
                        } else {
#pragma unroll
                            for (int e = 0; e < W; ++e) x.v[e] = x.v[e] + al * p.v[e];
                        }
                    }
                    Vec<ST, W> us = vload<ST, W>(U + o);
                    Vec<KT, W> op;
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        if constexpr (DF) {
                            us.v[e] = df_add(us.v[e], x.v[e]);
                            // within ulp(op) / 2 of u_j + delta
                            op.v[e] = dvalid ? us.v[e].x + (us.v[e].y + x.v[e]) : us.v[e].x;
                        } else {
                            us.v[e] += x.v[e];
                            op.v[e] = us.v[e];
                        }
                    }
                    if (DF && dvalid) vstore(X + o, x);
                    vstore(U + o, us);
                    vstore(T + own + o, op);
                    push(Tb, Ta, o, op);
                    if (snap_j || last) {
                        Vec<double, W> sd;
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            if constexpr (DF) sd.v[e] = df_value_bits(us.v[e].x, us.v[e].y);
                            else sd.v[e] = us.v[e];
                        }
                        if (snap_j) vstore(snap_j + o, sd);
                        if (last) vstore(outp + o, sd);
                    }
                }
            }
            // a non-finite state would only propagate: skip the remaining steps
            if (status == DERR_NONFINITE) break;
        }
        if (rank == 0 && tid == 0) {
            J.status[lb] = sh.status;
            J.its_total[lb] = (int)its_total;
            J.its_max[lb] = its_max;
        }
        __syncthreads();   // the next item resets sh.status and rewrites the tables
    }
    chip_cluster_sync();   // no CTA leaves while a neighbour may still store into its ghost planes
}

using ChipFn = void (*)(FineArgs, ChipPlan);
static void chip_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int C, int ctas, int threads, size_t smem,
                        cudaStream_t st) {
    cfg->gridDim = dim3((unsigned)ctas);
    cfg->blockDim = dim3((unsigned)threads);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
}
static ChipFn chip_fn(bool fp32, int n, bool pert) {
    if (!fp32) return pert ? fine_chip_kernel<double, 1, true> : fine_chip_kernel<double, 1, false>;
    if (n % 4 == 0) return pert ? fine_chip_kernel<float, 4, true> : fine_chip_kernel<float, 4, false>;
    return pert ? fine_chip_kernel<float, 1, true> : fine_chip_kernel<float, 1, false>;
}

// Shared memory of a CTA in a cluster of C, and which own-point vectors it holds; 0: too large.
static size_t chip_smem(int n, bool fp32, int C, int* keep) {
    const size_t n2 = (size_t)n * n, npl = (n + C - 1) / C, k = fp32 ? 4 : 8, st = 8;
    size_t bytes = (4 * (npl + 2) + 2) * n2 * k;
    bytes += (2 * npl * n + n2) * k * (fp32 ? 1 : 2);
    if (bytes > CHIP_SMEM) return 0;
    *keep = 0;
    const int bit[4] = {CHIP_U, CHIP_X, CHIP_F, CHIP_RH};
    const size_t word[4] = {st, k, k, k};
    for (int i = 0; i < 4; ++i) {
        const size_t need = npl * n2 * word[i];
        if (bytes + need <= CHIP_SMEM) {
            bytes += need;
            *keep |= bit[i];
        }
    }
    return bytes;
}

// Clusters of C CTAs that run at once with one CTA an SM (a GPC holds whole clusters only, so
// large ones leave SMs idle), asked of the driver once per device; 0: none fits, or no answer.
static int chip_clusters(int C) {
    static std::mutex mu;
    static std::vector<std::array<int, CHIP_MAXC + 1>> known;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    if ((int)known.size() <= dev) known.resize(dev + 1, std::array<int, CHIP_MAXC + 1>{});
    int& have = known[dev][C];
    if (have == 0) {
        ChipFn fn = chip_fn(false, 8, false);
        cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CHIP_SMEM);
        cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        chip_config(&cfg, at, C, C, 256, CHIP_SMEM, nullptr);
        int m = 0;
        if (cudaOccupancyMaxActiveClusters(&m, fn, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        have = std::max(0, m) + 1;
    }
    return have - 1;
}

// Whether a launch of B subintervals runs on chip, and in clusters of how many CTAs: the C of
// the least estimated time a step, if that is below the streaming kernels'.  The estimates (SM
// cycles) are fits to measured launches: a part for the barriers, reductions and scalars, and
// one for the points of a CTA's slab.  Against them, 40 steps, ms: FP64 (fine_kernel) 16^3 x 8
// 3.9 -> 1.24, 24^3 x 32 11.0 -> 4.2, 28^3 x 64 22.8 -> 14.3, but 32^3 x 64 25.0 -> 28.3 (three
// planes a CTA at most fit, so 11-CTA clusters in eight turns); FP32 16^3 x 16 1.27 -> 0.37
// (fine_kernel), 32^3 x 64 2.4 -> 1.5, 40^3 x 8 1.23 -> 0.75, but 40^3 x 64 2.8 -> 3.4 and
// 48^3 x 16 2.0 -> 2.3 (fused_kernel), 45^3 x 16 3.4 -> 2.5 (fine_kernel).
// A caller who fixes group_ctas gets that C whatever B, so that the result of a subinterval does not
// depend on how many share the launch: the nearest that fits on the grids where the cluster always
// wins, and on larger ones the other kernels where no cluster of that size fits.
bool fine_chip_plan(int n, bool fp32, int B, int group_ctas, ChipChoice* out) {
    if (n < 4) return false;
    const bool nearest = n <= (fp32 ? 36 : 28);
    double best = 0.0;
    out->C = 0;
    const double n2 = (double)n * n;
    const int cmax = std::min(n, CHIP_MAXC);
    for (int C = 1; C <= cmax; ++C) {
        int keep = 0;
        const size_t smem = chip_smem(n, fp32, C, &keep);
        if (smem == 0) continue;
        double t;
        if (group_ctas > 0 && !nearest && C != group_ctas) continue;
        const int at_once = chip_clusters(C);
        if (at_once == 0) continue;
        if (group_ctas > 0) {
            t = std::abs(C - group_ctas);
        } else {
            const double npl = (n + C - 1) / C;
            const double fix = fp32 ? 12000.0 : 28000.0;
            const double work = fp32 ? (n % 4 ? 6.0 : 2.7) * n2 * (npl + 0.7) : 70.0 * n2 * npl;
            // clusters in turn, or two an SM where they fit: those share its pipes
            const int deep = (B + at_once - 1) / at_once;
            if (smem > CHIP_SMEM / 2 || deep == 1) t = deep * (fix + work);
            else t = (deep / 2) * (fix + 2.0 * work) + (deep % 2) * (fix + work);
        }
        if (out->C == 0 || t < best) {
            best = t;
            out->C = C;
            out->keep = keep;
            out->smem = smem;
        }
    }
    if (out->C == 0) return false;
    if (group_ctas > 0) return true;
    const double pts = B * n2 * n;
    const double streamed = fp32 ? (n % 4 ? 45000.0 + 0.11 * pts : 50000.0 + 0.023 * pts)
                                 : 150000.0 + (n % 4 ? 0.95 : 0.55) * pts;
    return best < streamed;
}

void fine_chip_groups(int n, bool fp32, int B, std::vector<int>* out) {
    ChipChoice ch;
    if (fine_chip_plan(n, fp32, B, 0, &ch)) out->push_back(ch.C);
    for (int C = 1, last = 0; C <= CHIP_MAXC; ++C) {   // the smallest cluster of each slab height
        if (!fine_chip_plan(n, fp32, B, C, &ch) || ch.C != C || (n + C - 1) / C == last) continue;
        last = (n + C - 1) / C;
        out->push_back(C);
    }
}

cudaError_t launch_fine_chip(const FineArgs& a, bool fp32, const ChipChoice& ch, int max_groups, cudaStream_t st) {
    const int n = a.g.n, W = fp32 && n % 4 == 0 ? 4 : 1;
    ChipPlan cp;
    cp.C = ch.C;
    cp.Cp = 1;
    while (cp.Cp < ch.C) cp.Cp *= 2;
    cp.npl = (n + ch.C - 1) / ch.C;
    cp.keep = ch.keep;
    const int lanes = n / W, npos = n * lanes;
    cp.mpos = (unsigned)((1ull << 32) / npos + 1);
    cp.mlane = lanes > 1 ? (unsigned)((1ull << 32) / lanes + 1) : 0u;
    ChipFn fn = chip_fn(fp32, n, a.jobs[0].pert != nullptr);
    const int units = cp.npl * npos;
    int thr = fp32 ? 512 : 256;   // FP64: two warps a sub-partition keep its pipe busy (512: 10 % slower)
    while (thr > 128 && thr / 2 >= units) thr /= 2;
    cudaError_t e = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CHIP_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    chip_config(&cfg, at, ch.C, std::min(a.B, max_groups) * ch.C, thr, ch.smem, st);
    e = cudaLaunchKernelEx(&cfg, fn, a, cp);
    ++g_launch_count;
    return e;
}

}  // namespace pr
