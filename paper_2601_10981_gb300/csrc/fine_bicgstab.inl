// BiCGStab iterations it + 1, it + 2, ... of one step from the residual r (rhat in rh) until it
// stops; `first` iterations take p from r.  Uses the lambdas of fine_march.inl and finish();
// returns from the enclosing function with FINE_GIVE_UP when a barrier gives up.  FINE_PIPE: the
// marches load a plane ahead into registers.
            while (!conv) {
                ++it;
                // ---------------- ph1: p = r + beta (p' - omega v'), v = A p
                KT* pn = (it & 1) ? p1 : p0;
                KT* po = (it & 1) ? p0 : p1;
                KT* vn = (it & 1) ? v1 : v0;
                KT* vo = (it & 1) ? v0 : v1;
                {
                    const KT bk = (KT)sh.beta, ok = (KT)sh.omega;
                    const bool first = (it == 1);
                    Acc<KT, 1> acc;
                    acc.init();
                    march(FINE_PIPE, ringk,
                          [&](int i) -> RawP<KT, W> {
                              RawP<KT, W> o;
                              o.r = vload<KT, W>(r + i);
                              if (!first) {
                                  o.p = vload<KT, W>(po + i);
                                  o.v = vload<KT, W>(vo + i);
                              } else {
#pragma unroll
                                  for (int e = 0; e < W; ++e) { o.p.v[e] = (KT)0; o.v.v[e] = (KT)0; }
                              }
                              return o;
                          },
                          [&](const RawP<KT, W>& v) -> VK {
                              VK o;
#pragma unroll
                              for (int e = 0; e < W; ++e) o.v[e] = v.r.v[e] + bk * (v.p.v[e] - ok * v.v.v[e]);
                              return o;
                          },
                          [&](int i) -> OwnH<KT, W, PT> { return {vload<KT, W>(rh + i), {}}; },
                          [&](int i, int k, int, const OwnH<KT, W, PT>& ow, const KT* rowc, const KT* rowzp,
                              const KT* rowzm) {
                              const VK& rhv = ow.h;
                              const auto q7 = nb7(rowc, rowzp, rowzm);
                              const VK av = applyA(k, q7.c, q7.xp, q7.xm, q7.yp, q7.ym, q7.zp, q7.zm, load_pert(i));
                              vstore(pn + i, q7.c);
                              vstore(vn + i, av);
#pragma unroll
                              for (int e = 0; e < W; ++e) acc.f[0] += rhv.v[e] * av.v[e];
                              acc.tick();
                          });
                    if (!finish(acc, [&](const double* s) {
                    const double rv = s[0];
                    if (rv == 0.0 || !isfinite(rv)) {
                        sh.status = isfinite(rv) ? DERR_BREAKDOWN : DERR_NONFINITE;
                        sh.flag = 1;
                    } else {
                        sh.alpha = sh.rho / rv;
                        sh.flag = 0;
                    }
                    })) return FINE_GIVE_UP;
                }
                if (sh.flag) {
                    --it;
                    break;
                }
                // ---------------- ph2: s = r - alpha v, t = A s
                {
                    const KT al = (KT)sh.alpha;
                    Acc<KT, 3> acc;
                    acc.init();
                    march(FINE_PIPE, ringk,
                          [&](int i) -> RawS<KT, W> { return {vload<KT, W>(r + i), vload<KT, W>(vn + i)}; },
                          [&](const RawS<KT, W>& v) -> VK {
                              VK o;
#pragma unroll
                              for (int e = 0; e < W; ++e) o.v[e] = v.r.v[e] - al * v.v.v[e];
                              return o;
                          },
                          [&](int) -> NoOwn { return NoOwn{}; },
                          [&](int i, int k, int, const NoOwn&, const KT* rowc, const KT* rowzp,
                              const KT* rowzm) {
                              const auto q7 = nb7(rowc, rowzp, rowzm);
                              const VK tv = applyA(k, q7.c, q7.xp, q7.xm, q7.yp, q7.ym, q7.zp, q7.zm, load_pert(i));
                              vstore(t + i, tv);
#pragma unroll
                              for (int e = 0; e < W; ++e) {
                                  acc.f[0] += tv.v[e] * q7.c.v[e];
                                  acc.f[1] += tv.v[e] * tv.v[e];
                                  acc.f[2] += q7.c.v[e] * q7.c.v[e];
                              }
                              acc.tick();
                          });
                    if (!finish(acc, [&](const double* s) {
                    const double ts = s[0], tt2 = s[1], ss = s[2];
                    const int half = sqrt(ss) <= sh.thr;
                    if (!half) {
                        if (tt2 == 0.0 || !isfinite(tt2)) {
                            sh.status = isfinite(tt2) ? DERR_BREAKDOWN : DERR_NONFINITE;
                            sh.omega = 0.0;
                        } else {
                            sh.omega = ts / tt2;
                            if (sh.omega == 0.0) sh.status = DERR_BREAKDOWN;
                        }
                    }
                    sh.flag = half;
                    })) return FINE_GIVE_UP;
                }
                const bool half = sh.flag != 0;
                // ---------------- ph3: delta += alpha p + omega s ; r = s - omega t
                {
                    const KT al = (KT)sh.alpha, om = (KT)sh.omega;
                    const bool first = (it == 1) && !xg;   // delta holds the initial guess
                    const bool upd_r = !half && sh.status == 0;
                    Acc<KT, 2> acc;
                    acc.init();
                    // the update of the owned points from their six inputs
                    auto p3_fn = [&](int i, const Raw6<KT, W>& v) {
                        VK dn, rn;
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            const KT sc_ = v.r.v[e] - al * v.v.v[e];
                            dn.v[e] = v.d.v[e] + al * v.p.v[e] + om * sc_;
                            rn.v[e] = sc_ - om * v.t.v[e];
                            acc.f[0] += v.h.v[e] * rn.v[e];
                            acc.f[1] += rn.v[e] * rn.v[e];
                        }
                        vstore(delta + i, dn);
                        vstore(rw + i, rn);
                        acc.tick();
                    };
                    bool staged3 = false;
                    if constexpr (DF && KS == 1) {
                        if (upd_r) {
                            // inputs of plane z staged by cp.async while planes z-2, z-1 are
                            // updated; each thread reads back only what it copied, so no
                            // barrier is needed; layout [slot][input][thread][W] (no bank
                            // conflicts).  The ring is idle in this phase.
                            staged3 = true;
                            constexpr int NS = FINE_PH3_SLOTS;
                            float* stg = reinterpret_cast<float*>(ring_raw);
                            const int nthr = blockDim.x;
                            const bool act = ty < TY;
                            auto sad = [&](int sl, int q) { return stg + ((size_t)(sl * 6 + q) * nthr + threadIdx.x) * W; };
                            for (int tt = t_lo; tt < t_hi; ++tt) {
                                int y0, zlo, zhi;
                                geo.tile(tt, y0, zlo, zhi);
                                const int rowoff = (y0 + ty) * n + x0;
                                auto issue = [&](int z, int sl) {
                                    if (act && z < zhi) {
                                        const long long i = (long long)z * n2 + rowoff;
                                        if (!first) cp_async_b<4 * W>(sad(sl, 0), delta + i);
                                        cp_async_b<4 * W>(sad(sl, 1), pn + i);
                                        cp_async_b<4 * W>(sad(sl, 2), r + i);
                                        cp_async_b<4 * W>(sad(sl, 3), vn + i);
                                        cp_async_b<4 * W>(sad(sl, 4), t + i);
                                        cp_async_b<4 * W>(sad(sl, 5), rh + i);
                                    }
                                    cp_async_commit_group();
                                };
#pragma unroll
                                for (int d = 0; d < NS - 1; ++d) issue(zlo + d, d);
                                int sl = 0;
                                for (int z = zlo; z < zhi; ++z) {
                                    // refill the slot of plane z - 1 (read last iteration)
                                    issue(z + NS - 1, sl == 0 ? NS - 1 : sl - 1);
                                    cp_async_wait_newest<NS - 1>();
                                    if (act) {
                                        Raw6<KT, W> v;
                                        if (!first) v.d = vload<float, W>(sad(sl, 0));
                                        else {
#pragma unroll
                                            for (int e = 0; e < W; ++e) v.d.v[e] = 0.0f;
                                        }
                                        v.p = vload<float, W>(sad(sl, 1));
                                        v.r = vload<float, W>(sad(sl, 2));
                                        v.v = vload<float, W>(sad(sl, 3));
                                        v.t = vload<float, W>(sad(sl, 4));
                                        v.h = vload<float, W>(sad(sl, 5));
                                        p3_fn(z * n2 + rowoff, v);
                                    }
                                    sl = (sl + 1 == NS) ? 0 : sl + 1;
                                }
                                cp_async_wait_newest<0>();
                            }
                        }
                    }
                    if (upd_r && !staged3) {
                        owned([&](int i) -> Raw6<KT, W> {
                                  Raw6<KT, W> o;
                                  if (!first) o.d = vload<KT, W>(delta + i);
                                  else {
#pragma unroll
                                      for (int e = 0; e < W; ++e) o.d.v[e] = (KT)0;
                                  }
                                  o.p = vload<KT, W>(pn + i);
                                  o.r = vload<KT, W>(r + i);
                                  o.v = vload<KT, W>(vn + i);
                                  o.t = vload<KT, W>(t + i);
                                  o.h = vload<KT, W>(rh + i);
                                  return o;
                              },
                              p3_fn);
                    } else if (!upd_r) {
                        owned([&](int i) -> RawP2<KT, W> {
                                  RawP2<KT, W> o;
                                  if (!first) o.d = vload<KT, W>(delta + i);
                                  else {
#pragma unroll
                                      for (int e = 0; e < W; ++e) o.d.v[e] = (KT)0;
                                  }
                                  o.p = vload<KT, W>(pn + i);
                                  return o;
                              },
                              [&](int i, const RawP2<KT, W>& v) {
                                  VK dn;
#pragma unroll
                                  for (int e = 0; e < W; ++e) dn.v[e] = v.d.v[e] + al * v.p.v[e];
                                  vstore(delta + i, dn);
                              });
                    }
                    if (!finish(acc, [&](const double* s) {
                        if (!upd_r) return;   // delta is final
                        const double rho_new = s[0], rr1 = s[1];
                        int stop = 1;
                        if (!isfinite(rr1)) sh.status = DERR_NONFINITE;
                        else if (sqrt(rr1) <= sh.thr) {}
                        else if (rho_new == 0.0) sh.status = DERR_BREAKDOWN;
                        else if (it >= J.maxit) sh.status = DERR_NOT_CONVERGED;
                        else {
                            sh.beta = (rho_new / sh.rho) * (sh.alpha / sh.omega);
                            sh.rho = rho_new;
                            stop = 0;
                        }
                        sh.flag = stop;
                    })) return FINE_GIVE_UP;
                    if (!upd_r) break;
                    r = rw;
                }
                if (sh.flag) break;
            }
