// Batched symmetric eigensolver of the POD and the selection of Algorithm 1: eigenpairs of each
// Gram matrix, numerical rank, dimension m, and C = Y_m Lambda_m^{-1/2}.
//
// Parallel cyclic Jacobi in FP64 (round-robin pairing).  One round rotates K/2 disjoint pairs:
// A <- J^T A J, V <- V J.  GB300 retires 2 FP64 operations a cycle and SM, so a round of a 64 x 64
// matrix is 12,000 cycles of one SM's FP64 pipe beside a chain of divisions and square roots
// (560 to 690 cycles each) for the angles and two barriers between passes; with one CTA a matrix
// a handful of windows left the chip idle.  Here
//   * a thread-block cluster of C CTAs works on a matrix, each on the rows of its pairs ("slots")
//     of A and on a share of V's rows;
//   * A is kept in the order of the pairing: rows and columns 2 i, 2 i + 1 are slot i's p and q,
//     and the 2 x 2 block of two slots gets both its rotations from a pair of lanes in registers.
//     Between rounds the players move one slot on, so a block's results go to the other buffer
//     at the next round's places, the ones that change hands into the neighbour CTA's memory;
//   * the three entries an angle needs go to every CTA as they are formed, and after the one
//     cluster barrier of a round each CTA forms all angles for itself (a warp needs the same time
//     for 1 pair and for 32) while its other warps, on the other three sub-partitions, update V;
//   * the angle starts from an FP32 estimate of tan and takes one Newton step in FP64, and the
//     cosine one third-order step of the inverse square root (Householder's iteration), ten FP64
//     operations deep in place of four divisions and roots.
// POD of 64 windows of 32 snapshots on 64^3 (C = 2): 11.1 -> 9.7 ms, the solver 3.3 ms of it before;
// of four windows of 64 on 128^3 (C = 8): 27.2 -> 18.2 ms, the solver 12.1 ms of it before.
// A round takes 5,100 cycles (K = 32, C = 2 or K = 64, C = 8; about 12,000 at K = 64 before): 2,500
// to 3,400 for the blocks, 400 to 900 to arrive at the barrier, 1,900 for the angles.
#include "df.cuh"
#include "pr_internal.cuh"

#include <algorithm>
#include <math.h>

namespace pr {

constexpr int EIG_THREADS = 256;
constexpr int EIG_WARPS = EIG_THREADS / 32;
constexpr int EIG_VTHREADS = EIG_THREADS - 64;   // warps 0 and 4 (one sub-partition) form the angles
constexpr int EIG_MAX_SWEEPS = 40;
constexpr int EIG_MAXC = 8;
constexpr size_t EIG_SMEM = 224 * 1024;

// Round r of the pairing of Kp = 2 np players (Kp - 1 of them on a circle, the last one fixed):
// the players of slot i.
__device__ __forceinline__ void rr_pair(int r, int i, int Kp, int& p, int& q) {
    const int M = Kp - 1;
    p = r + i;
    q = r - i;
    if (p >= M) p -= M;
    if (q < 0) q += M;
    if (i == 0) p = M;
}
// Place (2 slot + role) in the next round of the player at place pos in this one.
__device__ __forceinline__ int rr_next(int pos, int np) {
    const int i = pos >> 1;
    if (np == 1) return pos;
    if (pos & 1) return i == np - 1 ? 2 * i : 2 * (i + 1) + 1;
    return i == 0 ? 0 : i == 1 ? 1 : 2 * (i - 1);
}

__device__ __forceinline__ void eig_cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void eig_cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ double* eig_peer(double* p, int rank) {
    unsigned long long o;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(o) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<double*>(o);
}

// double -> float on the integer pipe (conversions occupy the FP64 pipe), cut
__device__ __forceinline__ float eig_d2f(double x) { return d2df_bits(x).x; }

// The rotation that annihilates a_pq: t = tan solves a_pq t^2 + (a_qq - a_pp) t - a_pq = 0 (the
// smaller root).  Entries are scaled to below 2; one too small for a float (2^-126) stays.
__device__ __forceinline__ void eig_angle(double app, double apq, double aqq, double& c, double& s) {
    c = 1.0;
    s = 0.0;
    const float bf = eig_d2f(apq);
    if (bf == 0.0f) return;
    const double d = aqq - app;
    const float df = eig_d2f(d);
    const float tau = df / (2.0f * bf);
    const float t0 = (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
    double t = f2d_bits(t0);
    const double f = fma(apq, fma(t, t, -1.0), d * t);
    t -= f2d_bits(eig_d2f(f) / (2.0f * bf * t0 + df));
    const double w = fma(t, t, 1.0);
    const double y = f2d_bits(rsqrtf(eig_d2f(w)));
    const double e = fma(-(w * y), y, 1.0);
    c = fma(y * e, fma(0.375, e, 0.5), y);   // w^-1/2 to e^3, e < 2^-20
    s = t * c;
}

__host__ __device__ __forceinline__ size_t eig_doubles(int Kp, int C) {
    const int np = Kp / 2, nsl = (np + C - 1) / C, nv = (Kp + C - 1) / C;
    return (size_t)4 * nsl * Kp + (size_t)(nv * (Kp + 1) + 1) / 2 * 2 + 4 * np + 6 * np + 4 * Kp;
}
static size_t eig_smem(int Kp, int C) { return eig_doubles(Kp, C) * sizeof(double) + (size_t)Kp * sizeof(int); }

__global__ void __launch_bounds__(EIG_THREADS) eig_pod_kernel(EigArgs a, int C) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = blockIdx.x / C, rank = blockIdx.x % C;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = a.K[b];
    double* lam_out = a.lam + (size_t)b * a.maxK;
    double* Cb = a.C + (size_t)b * a.ldC_b;
    if (K <= 0) {   // the whole cluster leaves
        if (rank == 0 && tid == 0) a.m[b] = 0;
        return;
    }
    const int Kp = K + (K & 1), np = Kp / 2, M = Kp - 1;
    const int nsl = (np + C - 1) / C, s0 = min(rank * nsl, np), ns = min(nsl, np - s0);
    const int nv = (Kp + C - 1) / C, k0 = min(rank * nv, Kp), nk = min(nv, Kp - k0);
    const int ldv = Kp + 1;   // odd stride in doubles: V's column walks hit distinct banks
    double* A0 = reinterpret_cast<double*>(smem_raw);   // [2][2 nsl][Kp]
    double* V = A0 + (size_t)4 * nsl * Kp;              // [nv][ldv], by player
    double2* cs = reinterpret_cast<double2*>(V + (size_t)(nv * ldv + 1) / 2 * 2);   // [2][np]
    double* nd = reinterpret_cast<double*>(cs + 2 * np);   // [2][np][3]: a_pp, a_pq, a_qq
    double* lam = nd + 6 * np;                          // [Kp]
    double* sq = lam + Kp;                              // [Kp]
    double* red = sq + Kp;                              // [Kp][2]: a row's off-diagonal and diagonal squares
    int* perm = reinterpret_cast<int*>(red + 2 * Kp);   // [Kp]
    __shared__ int s_stop, s_e, s_r, s_m;
    const double* Gb = a.G + (size_t)b * a.ldG_b;

    // power-of-two scale: the largest entry into [1, 2) (exact, undone on the eigenvalues)
    if (tid == 0) s_e = s_r = 0;
    __syncthreads();
    int emax = 0;
    for (int e = tid; e < K * K; e += EIG_THREADS) {
        const int i = e / K, j = e - i * K;
        emax = max(emax, (__double2hiint(Gb[(size_t)i * a.ldG + j]) >> 20) & 0x7ff);
    }
    for (int o = 16; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if (lane == 0) atomicMax(&s_e, emax);
    __syncthreads();
    emax = s_e;
    if (emax == 0 || emax == 0x7ff) emax = 1023;
    const double scale = __hiloint2double(max(1, 2046 - emax) << 20, 0);
    const double unscale = __hiloint2double((2046 - max(1, 2046 - emax)) << 20, 0);

    auto entry = [&](int i, int j) { return i < K && j < K ? Gb[(size_t)i * a.ldG + j] * scale : 0.0; };
    for (int e = tid; e < 2 * ns * Kp; e += EIG_THREADS) {
        const int lr = e / Kp, pc = e - lr * Kp, pr = 2 * s0 + lr;
        int ip, iq, jp, jq;
        rr_pair(0, pr >> 1, Kp, ip, iq);
        rr_pair(0, pc >> 1, Kp, jp, jq);
        A0[e] = entry(pr & 1 ? iq : ip, pc & 1 ? jq : jp);
    }
    for (int e = tid; e < nk * Kp; e += EIG_THREADS) {
        const int k = e / Kp, j = e - k * Kp;
        V[k * ldv + j] = (k0 + k == j) ? 1.0 : 0.0;
    }
    for (int i = tid; i < np; i += EIG_THREADS) {
        int p, q;
        rr_pair(0, i, Kp, p, q);
        nd[3 * i] = entry(p, p);
        nd[3 * i + 1] = entry(p, q);
        nd[3 * i + 2] = entry(q, q);
    }
    auto cluster_sync = [&]() {
        if (C > 1) {
            eig_cluster_arrive();
            eig_cluster_wait();
        } else {
            __syncthreads();
        }
    };
    cluster_sync();   // every CTA has started, its memory may be written

    // angles of the round whose entries are in buffer w, by warps 0 and 4
    auto angles = [&](int w) {
        const int i = (warp >> 2) * 32 + lane;
        if ((warp & 3) == 0 && i < np) {
            double c = 1.0, s = 0.0;
            const double* x = nd + 3 * (w * np + i);
            if (i != 0 || !(K & 1)) eig_angle(x[0], x[1], x[2], c, s);   // slot 0 of an odd K rests
            cs[w * np + i] = make_double2(c, s);
        }
    };
    angles(0);
    // fixed shares: lanes l and l + 16 hold a block of A (its rows p and q, then its columns)
    const int h = lane >> 4, units = ns * np;
    const int u0 = warp * 16 + (lane & 15), ustep = EIG_WARPS * 16;
    const int ui0 = u0 / np, uj0 = u0 - ui0 * np, udi = ustep / np, udj = ustep - udi * np;
    const int vt = (warp < 4 ? warp - 1 : warp - 2) * 32 + lane;
    const bool vwarp = (warp & 3) != 0;
    const int vk0 = vt / np, vi0 = vt - vk0 * np, vdk = EIG_VTHREADS / np, vdi = EIG_VTHREADS - vdk * np;
    int cur = 0;
    double prev = 0.0;
    __syncthreads();
    for (int sweep = 0; sweep < EIG_MAX_SWEEPS; ++sweep) {
        // convergence: off-diagonal Frobenius norm against the whole matrix
        {
            const double* A = A0 + (size_t)cur * 2 * nsl * Kp;
            // row by row, eight lanes a row, then the rows in a fixed order: the same sums, and so
            // the same rotations, for every C (which follows the number of matrices in the launch)
            for (int l0 = 0; l0 < 2 * ns; l0 += EIG_THREADS / 8) {
                const int lr = l0 + (tid >> 3), pr = 2 * s0 + lr;
                double off = 0.0;
                if (lr < 2 * ns)
                    for (int pc = tid & 7; pc < Kp; pc += 8) {
                        const double v = A[lr * Kp + pc];
                        if (pc != pr) off = fma(v, v, off);
                    }
                for (int o = 4; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
                if (lr < 2 * ns && (tid & 7) < C) {
                    const double v = A[lr * Kp + pr];
                    double* r = C > 1 ? eig_peer(red, tid & 7) : red;
                    r[2 * pr] = off;
                    r[2 * pr + 1] = v * v;
                }
            }
            cluster_sync();
            if (warp == 0) {
                double off = 0.0, dia = 0.0;
                for (int i = lane; i < Kp; i += 32) {
                    off += red[2 * i];
                    dia += red[2 * i + 1];
                }
                for (int o = 16; o > 0; o >>= 1) {
                    off += __shfl_xor_sync(0xffffffffu, off, o);
                    dia += __shfl_xor_sync(0xffffffffu, dia, o);
                }
                // converged when the off-diagonal part is at the rounding level of the Gram
                // matrix itself, ||off||_F <= K eps ||A||_F: a tighter bound sits below the
                // noise of the rotations (fused multiply-adds) and would never be met.  The
                // rotations' own noise can also sit just above that bound, so a sweep that no
                // longer cuts ||off|| four-fold within 16 times of it ends the iteration too
                // (past the quadratic phase further sweeps only reshuffle rounding noise).
                // Every CTA adds the same numbers in the same order and decides alike.
                const double tot = off + dia, tolK = (double)K * 2.220446049250313e-16;
                const double lim = tolK * tolK * tot;
                const bool stalled = sweep > 0 && off <= 256.0 * lim && off * 16.0 >= prev;
                if (lane == 0) s_stop = off <= lim || tot == 0.0 || stalled;
                prev = off;
            }
            __syncthreads();
            if (s_stop) break;
        }
        for (int r = 0; r < M; ++r) {
            const int nxt = cur ^ 1;
            const double2* csr = cs + cur * np;
            {   // A <- J^T A J
                const double* A = A0 + (size_t)cur * 2 * nsl * Kp;
                double* An = A0 + (size_t)nxt * 2 * nsl * Kp;
                double* ndn = nd + 3 * nxt * np;
                int i = ui0, j = uj0;
                for (int base = warp * 16; base < units; base += ustep) {
                    const bool act = i < ns;
                    double y0 = 0.0, y1 = 0.0;
                    double2 ci = make_double2(1.0, 0.0);
                    if (act) {
                        const double2 x = *reinterpret_cast<const double2*>(A + (2 * i + h) * Kp + 2 * j);
                        const double2 cj = csr[j];
                        ci = csr[s0 + i];
                        y0 = cj.x * x.x - cj.y * x.y;
                        y1 = cj.y * x.x + cj.x * x.y;
                    }
                    const double o = __shfl_xor_sync(0xffffffffu, h ? y0 : y1, 16);
                    if (act) {
                        const double a0 = h ? o : y0, a1 = h ? y1 : o;
                        const double z[2] = {ci.x * a0 - ci.y * a1, ci.y * a0 + ci.x * a1};
                        const int pc = rr_next(2 * j + h, np);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int pr = rr_next(2 * (s0 + i) + e, np), sl = pr >> 1;
                            const int to = sl < s0 ? rank - 1 : sl >= s0 + nsl ? rank + 1 : rank;
                            double* dst = An + (pr - 2 * to * nsl) * Kp + pc;
                            if (to != rank) dst = eig_peer(dst, to);
                            *dst = z[e];
                            if (sl == (pc >> 1) && !((pr & 1) && !(pc & 1))) {
                                double* x = ndn + 3 * sl + (pr & 1) + (pc & 1);
                                if (C == 1) *x = z[e];
                                else for (int k = 0; k < C; ++k) *eig_peer(x, k) = z[e];
                            }
                        }
                    }
                    i += udi;
                    j += udj;
                    if (j >= np) { j -= np; ++i; }
                }
            }
            if (C > 1) eig_cluster_arrive(); else __syncthreads();
            if (vwarp) {   // V <- V J (columns p, q)
                int k = vk0, i = vi0;
                while (k < nk) {
                    int p, q;
                    rr_pair(r, i, Kp, p, q);
                    const double2 c = csr[i];
                    double* v = V + k * ldv;
                    const double vp = v[p], vq = v[q];
                    v[p] = c.x * vp - c.y * vq;
                    v[q] = c.y * vp + c.x * vq;
                    k += vdk;
                    i += vdi;
                    if (i >= np) { i -= np; ++k; }
                }
            }
            if (C > 1) eig_cluster_wait();
            angles(nxt);
            __syncthreads();
            cur = nxt;
        }
    }
    // eigenvalues, descending order (ties by index)
    for (int lr = tid; lr < 2 * ns; lr += EIG_THREADS) {
        const int pos = 2 * s0 + lr;
        int p, q;
        rr_pair(0, pos >> 1, Kp, p, q);
        const double v = A0[((size_t)cur * 2 * nsl + lr) * Kp + pos] * unscale + 0.0;
        for (int k = 0; k < C; ++k) (C > 1 ? eig_peer(lam, k) : lam)[pos & 1 ? q : p] = v;
    }
    cluster_sync();   // the last writes into another CTA's memory
    auto key = [&](int i) {   // ordered as the doubles are, NaN too
        const long long k = __double_as_longlong(lam[i]);
        return k < 0 ? k ^ 0x7fffffffffffffffLL : k;
    };
    for (int i = tid; i < K; i += EIG_THREADS) {
        int rk = 0;
        const long long li = key(i);
        for (int j = 0; j < K; ++j) {
            const long long lj = key(j);
            rk += (lj > li) || (lj == li && j < i);
        }
        perm[rk] = i;
    }
    __syncthreads();
    const double l1 = lam[perm[0]];
    for (int i = tid; i < K; i += EIG_THREADS) {
        const double l = lam[perm[i]];
        sq[i] = sqrt(l);
        if (l > a.tau * l1) atomicAdd(&s_r, 1);
    }
    __syncthreads();
    if (tid == 0) {
        int m = 0;
        if (l1 > 0.0) {
            const int r = s_r;
            double total = 0.0;
            for (int i = 0; i < r; ++i) total += sq[i];
            double cum = 0.0;
            m = r;
            for (int i = 0; i < r; ++i) {
                cum += sq[i];
                if (cum >= a.gamma * total) { m = i + 1; break; }
            }
            if (a.cap > 0) m = min(m, a.cap);
            m = min(m, r);
        }
        s_m = m;
        if (rank == 0) a.m[b] = m;
    }
    __syncthreads();
    if (rank == 0)
        for (int i = tid; i < a.maxK; i += EIG_THREADS) lam_out[i] = (i < K) ? lam[perm[i]] : 0.0;
    const int m = s_m, rows = min(nk, K - k0);
    for (int e = tid; e < rows * m; e += EIG_THREADS) {
        const int i = e / m, j = e - i * m;
        Cb[(size_t)(k0 + i) * a.ldC + j] = V[i * ldv + perm[j]] / sq[j];
    }
}

cudaError_t launch_eig_pod(const EigArgs& a, cudaStream_t st) {
    if (a.B <= 0) return cudaSuccess;
    const int Kp = std::max(2, a.maxK + (a.maxK & 1));
    if (Kp > 118) return cudaErrorInvalidValue;   // two full matrices within one CTA's shared memory
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(eig_pod_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_SMEM);
    if (e != cudaSuccess) return e;
    // The largest cluster whose CTAs get an SM each (clusters of 4 and 8 leave a few SMs of the
    // chip's processing clusters over) and hold four slots or more.
    int C = 1;
    for (int c = 2; c <= EIG_MAXC; c *= 2)
        if (eig_smem(Kp, C) > EIG_SMEM || (8 * c <= Kp && a.B <= sms / c - (c == 8 ? 4 : c == 4 ? 2 : 0))) C = c;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3((unsigned)(a.B * C));
    cfg.blockDim = dim3(EIG_THREADS);
    cfg.dynamicSmemBytes = eig_smem(Kp, C);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, eig_pod_kernel, a, C);
    ++g_launch_count;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace pr
