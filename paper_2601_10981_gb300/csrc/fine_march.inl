// The tile march, the pointwise loop and the operator of the streaming fine kernels, as lambdas
// over the thread's constants (included in the body of the functions that run a general
// BiCGStab iteration, so that they stay in registers there): W, KF, KS, PT, KT; n, n2, Ng, ty,
// x0, xl, xr, RP, TY, RW, geo, t_lo, t_hi; tabk, ky_x, kz_x, c0, c1, bpk, kp; ring_lo.
    KT kx_y[KS], kz_y[KS];
    KT kx_z = 0, ky_z = 0;
    auto tile_terms = [&](int y0) {
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int y = min(y0 + ty + k * RP, n - 1);
            kx_y[k] = tabk[TXY * n + y];
            kz_y[k] = tabk[TZY * n + y];
        }
    };
    auto plane_terms = [&](int z) {
        kx_z = tabk[TXZ * n + z];
        ky_z = tabk[TYZ * n + z];
    };

    // The x +- 1 neighbours of the W points: shifts of the centre vector plus one edge
    // value on each side read from the ring row.
    auto shift = [&](const auto* row, const auto& c, auto& xp, auto& xm) {
#pragma unroll
        for (int e = 0; e < W - 1; ++e) {
            xp.v[e] = c.v[e + 1];
            xm.v[e + 1] = c.v[e];
        }
        xp.v[W - 1] = row[xr];
        xm.v[0] = row[xl];
    };

    // ---- tile march for stencil phases (ring of FINE_SLOTS planes, one barrier per
    // FINE_PLANES planes):
    //   load(i) -> Raw            inputs of the operand at the W points from index i
    //   opnd(Raw) -> Vec          operand values written into the ring
    //   own(i) -> Own             inputs the output needs at owned points
    //   out(i, k, y, Own, rowc, rowzp, rowzm)   per owned W points (k: row slot); rowc is
    //                             the ring row of the points, rowzp / rowzm the rows above /
    //                             below in z; rowc +- n are the y neighbours
    // Plane p lives in slot (p - zlo + 1) mod FINE_SLOTS.  A round at z commits planes
    // z+1 .. z+np (np <= PL), then the barrier, then the stencils of planes z .. z+np-1
    // read planes z-1 .. z+np.  A thread that runs ahead can only reach the commits of
    // the next round, planes z+np+1 .. z+2np, whose slots differ from those of z-1 .. z+np
    // as long as 2 PL + 2 <= FINE_SLOTS; the next barrier stops it there.
    //   pipe                       true: prefetch the next round's first plane during the
    //                              stencils; false: load each plane just before committing
    //                              it (fewer live registers)
    auto march = [&](bool pipe, auto* ring, auto&& load, auto&& opnd, auto&& own, auto&& out) {
        using Raw = decltype(load(0));
        using Own = decltype(own(0));
        constexpr int PL = FINE_PLANES, NSL = FINE_SLOTS;
        for (int tt = t_lo; tt < t_hi; ++tt) {
            int y0, zlo, zhi;
            geo.tile(tt, y0, zlo, zhi);
            tile_terms(y0);
            int fidx[KF];
#pragma unroll
            for (int k = 0; k < KF; ++k) {
                const int rr = ty + k * RP;
                int y = y0 + rr - 1;
                y = (y < 0) ? y + n : (y >= n ? y - n : y);
                fidx[k] = (rr < RW) ? y * n + x0 : -1;   // in-plane offset, -1: no row
            }
            Raw pre[KF];
            Own opre[KS];
            auto prefetch = [&](int zp) {
                const int zz = (zp < 0) ? zp + n : (zp >= n ? zp - n : zp);
#pragma unroll
                for (int k = 0; k < KF; ++k)
                    if (fidx[k] >= 0) pre[k] = load(zz * n2 + fidx[k]);
            };
            auto own_of = [&](int z, Own (&dst)[KS]) {
#pragma unroll
                for (int k = 0; k < KS; ++k)
                    if (ty + k * RP < TY) dst[k] = own(z * n2 + (y0 + ty + k * RP) * n + x0);
            };
            auto slot = [&](int p) { return (p - zlo + 1) % NSL; };
            auto commit = [&](int sl) {
#pragma unroll
                for (int k = 0; k < KF; ++k) {
                    const int rr = ty + k * RP;
                    if (fidx[k] < 0) continue;
                    auto* dst = ring + (sl * RW + rr) * n + x0;
                    const auto val = opnd(pre[k]);
                    if constexpr (is_hilo<std::decay_t<decltype(val)>>::value) {
                        vstore(dst, val.hi);
                        vstore(dst + ring_lo, val.lo);
                    } else if constexpr (is_ophilo<std::decay_t<decltype(val)>>::value) {
                        vstore(dst, val.op);
                        vstore(dst + ring_lo, val.hi);
                        vstore(dst + 2 * ring_lo, val.lo);
                    } else {
                        vstore(dst, val);
                    }
                }
            };
            prefetch(zlo - 1);
            commit(0);
            prefetch(zlo);
            commit(1);
            if (pipe) {
                prefetch(zlo + 1);
                own_of(zlo, opre);
            }
            for (int z = zlo; z < zhi; z += PL) {
                const int np = min(PL, zhi - z);
#pragma unroll
                for (int q = 1; q <= PL; ++q) {
                    if (q > np) break;
                    if (!pipe || q > 1) prefetch(z + q);
                    commit(slot(z + q));
                }
                __syncthreads();
                Own cur[PL][KS];
                if (pipe) {
#pragma unroll
                    for (int k = 0; k < KS; ++k) cur[0][k] = opre[k];
#pragma unroll
                    for (int q = 1; q < PL; ++q)
                        if (q < np) own_of(z + q, cur[q]);
                    if (z + np < zhi) {
                        prefetch(z + np + 1);
                        own_of(z + np, opre);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < PL; ++q)
                        if (q < np) own_of(z + q, cur[q]);
                }
#pragma unroll
                for (int q = 0; q < PL; ++q) {
                    if (q >= np) break;
                    const int zq = z + q;
                    const int sc = slot(zq), sp = slot(zq + 1), sm = slot(zq - 1);
                    plane_terms(zq);
#pragma unroll
                    for (int k = 0; k < KS; ++k) {
                        const int rr = ty + k * RP;
                        if (rr >= TY) continue;
                        out(zq * n2 + (y0 + rr) * n + x0, k, y0 + rr, cur[q][k], ring + (sc * RW + rr + 1) * n,
                            ring + (sp * RW + rr + 1) * n, ring + (sm * RW + rr + 1) * n);
                    }
                }
            }
            __syncthreads();   // the next tile's prologue rewrites slots 0 and 1
        }
    };
    // ---- pointwise loop over owned points, one plane of KS rows at a time
    auto owned = [&](auto&& load, auto&& fn) {
        using Raw = decltype(load(0));
        for (int tt = t_lo; tt < t_hi; ++tt) {
            int y0, zlo, zhi;
            geo.tile(tt, y0, zlo, zhi);
            for (int z = zlo; z < zhi; ++z) {
                Raw v[KS];
#pragma unroll
                for (int k = 0; k < KS; ++k)
                    if (ty + k * RP < TY) v[k] = load(z * n2 + (y0 + ty + k * RP) * n + x0);
#pragma unroll
                for (int k = 0; k < KS; ++k)
                    if (ty + k * RP < TY) fn(z * n2 + (y0 + ty + k * RP) * n + x0, v[k]);
            }
        }
    };
    // The 7-point operand values of the W points from ring rows (vector loads).
    auto nb7 = [&](const auto* rowc, const auto* rowzp, const auto* rowzm) {
        using T = std::remove_const_t<std::remove_pointer_t<decltype(rowc)>>;
        Nb7<T, W> o;
        o.c = vload<T, W>(rowc + x0);
        shift(rowc, o.c, o.xp, o.xm);
        o.yp = vload<T, W>(rowc + n + x0);
        o.ym = vload<T, W>(rowc - n + x0);
        o.zp = vload<T, W>(rowzp + x0);
        o.zm = vload<T, W>(rowzm + x0);
        return o;
    };
    // The stored perturbation at the W points from index i (FINE_MODE_IMPLICIT_PERT).  It is
    // loaded where the stencil uses it, not one plane ahead with the other owned-point
    // inputs: its 3 W registers held across the march made the instantiation spill.
    auto load_pert = [&](int i) -> PertV<KT, W, PT> {
        PertV<KT, W, PT> o;
        if constexpr (PT) {
            o.x = vload<KT, W>(bpk + i);
            o.y = vload<KT, W>(bpk + Ng + i);
            o.z = vload<KT, W>(bpk + 2 * Ng + i);
        }
        return o;
    };
    // A = I + dt L at the W points of row slot k (pb: the perturbation there)
    auto applyA = [&](int k, const Vec<KT, W>& c, const Vec<KT, W>& xp, const Vec<KT, W>& xm,
                      const Vec<KT, W>& yp, const Vec<KT, W>& ym, const Vec<KT, W>& zp,
                      const Vec<KT, W>& zm, const PertV<KT, W, PT>& pb) -> Vec<KT, W> {
        Vec<KT, W> o;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            KT ax = kx_y[k] + kx_z;
            KT ay = ky_x[e] + ky_z;
            KT az = kz_x[e] + kz_y[k];
            if constexpr (PT) {
                ax += kp * pb.x.v[e];
                ay += kp * pb.y.v[e];
                az += kp * pb.z.v[e];
            }
            o.v[e] = c0 * c.v[e] + (ax - c1) * xp.v[e] - (ax + c1) * xm.v[e] + (ay - c1) * yp.v[e] -
                     (ay + c1) * ym.v[e] + (az - c1) * zp.v[e] - (az + c1) * zm.v[e];
        }
        return o;
    };
    using VK = Vec<KT, W>;
    using VD = Vec<double, W>;
