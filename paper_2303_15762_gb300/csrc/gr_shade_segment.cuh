// The shading of one path segment, included in the bodies of k_shade (all
// modes; WAVE) and k_paths (plain mode without next-event estimation; not
// WAVE).  It is text and not a function so that both kernels, and k_shade
// before and after k_paths existed, form the same fused multiply-adds: as an
// inlined function the same statements rounded differently, and images of
// k_shade changed in the last bits.
//
// The segment ended at hh (distance, leaf slot or -1): measurement on escape
// or at an emitter, else the interaction and the sampled child ray.  Names it
// uses: p, P, rows, tvals, V, S, slot, m, kk, seg, prev_delta, cls, pixel, Qv,
// smp, bin, gh, lambda, cstep, kw, s_ray2, and o, d, beta2, rho, T, xfv, pt, K,
// hq, want_shadow, want_density, which it changes.  It defines done: the
// sample has ended.  WAVE: the next segment's state goes to the slot; else it
// stays in o, d, beta2, rho, T, xfv.
  auto drop_companions = [&]() {
#pragma unroll
    for (int g = 0; g < 4; ++g)
      if (g != gh) hq[g] = 0.0f;
  };
  const int hslot = __float_as_int(hh.y);
  bool done = false;
  auto add_col = [&](float val) {
    pt.x += T[0][0] * val;
    if (NS == 4) {
      pt.y += T[1][0] * val;
      pt.z += T[2][0] * val;
      pt.w += T[3][0] * val;
    }
  };
  // a contribution to class member g: the hero's into the sample's own
  // sum, the others' straight into their range sums
  auto add_member = [&](int g, float val) {
    if (g == gh) {
      add_col(val);
      return;
    }
    member_add<NS>(P, (size_t)p.P, g, slot, T[0][0], NS == 4 ? T[1][0] : 0.0f, NS == 4 ? T[2][0] : 0.0f,
                   NS == 4 ? T[3][0] : 0.0f, val);
  };
  if (hslot < 0 && HERO) {
    // escape measured at every class wavelength, balance-heuristic weights
    float cf[4], den = 0.0f;
    class_shares(V, cls, Qv, cf);
#pragma unroll
    for (int g = 0; g < 4; ++g) den += cf[g] * hq[g];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float wq = cf[g] * hq[g];
      float val = 0.0f;
      if (wq > 0.0f) {
        const float mg = hero_escape_measure(S, d, step_lambda(V, cstep, cls + g * Qv), V.beta0);
        val = mg * (wq / den);
      }
      // a zero term leaves the member's sum as it is (the sums start at
      // +0 and a zero product cannot change them): no read-modify-write
      if (val != 0.0f) add_member(g, val);
    }
    done = true;
  } else if (hslot < 0 && ANISO) {
    float msum = 0.0f;
    for (int l = 0; l < S.n_lights; ++l) msum += measure_distant_aniso(S.lights[l], d, lambda, kw, K, xyz(xfv));
    add_col(msum);
    done = true;
  } else if (hslot < 0) {
    float msum = 0.0f;
    for (int l = 0; l < S.n_lights; ++l) {
      const gr_light L = S.lights[l];
      if (L.type == GR_LIGHT_ENV) {
        msum += L.E;
      } else {
        const float kap = 1.0f / (s_ray2 + src_spread2(lambda, L.coh_len_um));
        msum += L.E * vmf(d, f3(L.dir[0], L.dir[1], L.dir[2]), kap);
      }
    }
    add_col(msum);
    done = true;
  } else {
    const float t = hh.x;
    const float eta = xfv.w;  // |k| = eta k0 in the current medium
    footprint_update(t, kw * eta, beta2, rho);
    if (ANISO) {
      const float zb = t * 1e6f / (kw * eta);
      K.i11 += zb;
      K.i22 += zb;
    }
    const float3 x = o + t * d;
    const int mat = S.tri_mat[hslot];
    const gr_material M = S.mats[mat];
    if (M.type == GR_MAT_EMITTER && HERO) {
      // the hit measured at every class wavelength with its footprint; with
      // NEE after a diffuse vertex, power heuristic over the (wavelength,
      // technique) pairs: cf_j qpre_j p_{j,lobe} = cf_j q_j pb, cf_j qpre_j
      // p_{j,emitter}; else balance over the wavelengths
      const int ei = S.emitter_of_mat[mat];
      const float4 u = rng4(p.seed, V.view_index, pixel, smp, seg, kCallEmitFoot);
      const bool two = (p.flags & GR_FLAG_NEE) && !prev_delta && S.n_emitters > 0;
      float cf[4], qp[4] = {1.0f, 1.0f, 1.0f, 1.0f}, pb = 0.0f, den = 0.0f;
      class_shares(V, cls, Qv, cf);
      const float3 ne = emitter_normal(S, ei);
      if (two) {
        const float4 mi = P.mis[slot];  // (r2, g, kl2, cos) of the rough vertex that sampled d
        pb = rough_density(mi.y, mi.z, mi.x) * mi.w;
        const float4 q4 = P.hqp[slot];
        qp[0] = q4.x, qp[1] = q4.y, qp[2] = q4.z, qp[3] = q4.w;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (two) {
          const float lj = step_lambda(V, cstep, cls + j * Qv), kj = 2.0f * kPi * __frcp_rn(lj);
          const float kap = 1.0f / (1.0f / (2.0f * V.beta0 * V.beta0 * kj * kj) + src_spread2(lj, M.coh_len_um));
          const float a = cf[j] * hq[j] * pb, b = cf[j] * qp[j] * vmf(-d, ne, kap) / (float)S.n_emitters;
          den += a * a + b * b;
        } else {
          den += cf[j] * hq[j];
        }
      }
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        if (!(cf[g] * hq[g] > 0.0f) || !(den > 0.0f)) continue;
        const float lg = step_lambda(V, cstep, cls + g * Qv);
        float fbg = beta2, frg = rho;  // the member's footprint at the hit
        if (g != gh) member_footprint(rho, lg * __frcp_rn(lambda), V.beta0 * V.beta0, fbg, frg);
        const float mg = hero_measure_emitter(S, ei, x, d, fbg, frg, 2.0f * kPi * __frcp_rn(lg), lg, u.x, u.y);
        const float w = two ? cf[g] * cf[gh] * hq[g] * pb * pb / den : cf[g] * hq[g] / den;
        add_member(g, mg * w);
      }
      done = true;
    } else if (M.type == GR_MAT_EMITTER) {
      const int ei = S.emitter_of_mat[mat];
      float4 u = rng4(p.seed, V.view_index, pixel, smp, seg, kCallEmitFoot);
      float val = ANISO ? measure_emitter_aniso(S, ei, x, d, K, xyz(xfv), kw, lambda, u.x, u.y)
                        : measure_emitter(S, ei, x, d, beta2, rho, kw, lambda, u.x, u.y);
      float w = 1.0f;
      if (WAVE && (p.flags & GR_FLAG_NEE) && !prev_delta && S.n_emitters > 0 && val > 0.0f) {
        const float3 ne = emitter_normal(S, ei);
        const float kap = 1.0f / (s_ray2 + src_spread2(lambda, M.coh_len_um));
        const float pn = vmf(-d, ne, kap) / (float)S.n_emitters;
        const float4 mi = P.mis[slot];  // (r2, g, kl2, cos) of the rough vertex that sampled d
        const float pb = rough_density(mi.y, mi.z, mi.x) * mi.w;
        w = pb * pb / (pb * pb + pn * pn);
      }
      add_col(val * w);
      done = true;
    } else if (M.type == GR_MAT_ABSORBER || seg >= V.max_depth) {
      done = true;
    } else {
      if ((p.flags & GR_FLAG_RR) && seg >= 3) {
        const float q = fminf(1.0f, fmaxf(0.05f, T[0][0]));
        float4 u = rng4(p.seed, V.view_index, pixel, smp, seg, kCallRR);
        if (u.x >= q) {
          done = true;
        } else {
          const float iq = 1.0f / q;
          for (int r = 0; r < (NS == 1 ? 1 : 4); ++r)
            for (int c = 0; c < (NS == 1 ? 1 : 4); ++c) T[r][c] *= iq;
        }
      }
      if (!done) {
        // --- interaction with the reversed wavevector
        if (HERO) {
          // the density ratios before this vertex's decision and the
          // footprints at the vertex, for its next-event estimate and for
          // an emitter hit by the direction it samples
          // (the ratios are read only at a rough vertex's next-event
          // estimate and at an emitter hit after a diffuse rough lobe)
          if (M.type == GR_MAT_ROUGH) P.hqp[slot] = make_float4(hq[0], hq[1], hq[2], hq[3]);
        }
        const float4 v0 = __ldg(&S.tri[3 * hslot]), v1 = __ldg(&S.tri[3 * hslot + 1]),
                     v2 = __ldg(&S.tri[3 * hslot + 2]);
        float3 nrm = normalize(cross(xyz(v1) - xyz(v0), xyz(v2) - xyz(v0)));
        // the front (counter-clockwise) face looks outward (into air for a dielectric)
        const bool entering = !(dot(nrm, d) > 0.0f);
        if (!entering) nrm = -nrm;
        const float cos_i = -dot(d, nrm);
        const float4 u = rng4(p.seed, V.view_index, pixel, smp, seg, kCallLobe);
        FresnelM F{1.0f, 0.0f, 1.0f, 0.0f};
        bool refracted = false;
        float cos_t = 0.0f, n_rel = 1.0f, eta_next = eta;
        if (M.type == GR_MAT_DIELECTRIC) {
          const float eta_m = M.n_re + M.cauchy_b_um2 / (lambda * lambda);
          n_rel = entering ? eta_m : 1.0f / eta_m;
          F = dielectric_pick(cos_i, n_rel, u.x, refracted, cos_t);
          if (refracted) eta_next = entering ? eta_m : 1.0f;
        } else if (M.fresnel == 1) {
          F = fresnel_conductor(cos_i, M.n_re, M.n_im);
        }
        float cn[4];
        float3 s_o = f3(0.f, 0.f, 0.f);
        if (NS == 1) {
          T[0][0] *= F.a;
          cn[0] = T[0][0];
          if (ANISO) s_o = s_vector(nrm, -d, xyz(xfv));
        } else {
          const float3 k_o = -d;
          const float3 xf = xyz(xfv);
          s_o = s_vector(nrm, k_o, xf);
          const float3 p_o = cross(k_o, s_o);
          const float cphi = dot(xf, s_o), sphi = dot(xf, p_o);
          const float r2 = cphi * cphi + sphi * sphi;
          const float c2 = (cphi * cphi - sphi * sphi) / r2, s2 = 2.0f * cphi * sphi / r2;
          for (int r = 0; r < 4; ++r) {
            const float X0 = T[r][0], X3 = T[r][3];
            const float X1 = T[r][1] * c2 - T[r][2] * s2;
            const float X2 = T[r][1] * s2 + T[r][2] * c2;
            T[r][0] = F.a * X0 + F.b * X1;
            T[r][1] = F.b * X0 + F.a * X1;
            T[r][2] = F.cr * X2 - F.ci * X3;
            T[r][3] = F.ci * X2 + F.cr * X3;
            cn[r] = T[r][0];
          }
        }
        // --- sample the scattered distribution
        const float3 t_mir = d - dot(d, nrm) * nrm;
        float3 d_out = d;
        int delta = 1;
        float4 mis_rec = make_float4(0.0f, 0.0f, 1.0f, 0.0f);
        bool alive = true;
        float g_r = 0.0f;
        if (M.type == GR_MAT_GRATING) {
          float3 gt = f3(M.gdir[0], M.gdir[1], M.gdir[2]);
          gt = gt - dot(gt, nrm) * nrm;
          if (dot(gt, gt) < 1e-12f) {
            float3 e1, e2;
            onb(nrm, e1, e2);
            gt = e1;
          }
          gt = normalize(gt);
          const float step = lambda / M.period_um;
          const TableRow row = rows[V.table_base + mat * V.nb + bin];
          const int jm = row.jmax;
          const bool renorm = !(p.flags & GR_FLAG_NO_RENORM);
          // the table's pick; within its rounding of a CDF boundary the
          // FP32 copy decides, and within FP32's rounding FP64 does
          bool ambiguous;
          int pick = grating_pick_tab(jm, t_mir, step, gt, renorm, u.x, TableRound<TT>::rel, TableRound<TT>::abs,
                                      [&](int a) { return table_load<TT>(tvals, row.offset + a); }, ambiguous);
          if (ambiguous && sizeof(TT) != sizeof(float))
            pick = grating_pick_tab(jm, t_mir, step, gt, renorm, u.x, TableRound<float>::rel,
                                    TableRound<float>::abs,
                                    [&](int a) { return __ldg(p.table_vals32 + row.offset + a); }, ambiguous);
          if (ambiguous) {
            atomicAdd(&p.ctr->ref_lobe, 1ull);
            pick = grating_pick_fp64(bin_lambda_d(V, bin), M.height_um, jm, t_mir, step, gt, renorm, u.x,
                                     p.table_vals64 ? p.table_vals64 + row.offset : nullptr);
          }
          if (pick == 0x7fffffff) {
            alive = false;
          } else {
            const float3 tj = t_mir + ((float)pick * step) * gt;
            d_out = tj + sqrtf(fmaxf(0.0f, 1.0f - dot(tj, tj))) * nrm;
            if (HERO) {
              if (pick != 0) {
                drop_companions();  // the order's direction depends on the wavelength
              } else {
                // order 0 leaves in the same direction at every wavelength
                const float ph = order0_prob(row, t_mir, step, gt, renorm, p.table_vals32);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                  if (g == gh || hq[g] == 0.0f) continue;
                  const int bg = cls + g * Qv;
                  const float p0 = order0_prob(rows[V.table_base + mat * V.nb + bg], t_mir,
                                               bin_lambda(V, bg) / M.period_um, gt, renorm, p.table_vals32);
                  hq[g] = ph > 0.0f ? hq[g] * (p0 / ph) : 0.0f;
                }
              }
            }
          }
        } else if (M.type == GR_MAT_MIRROR) {
          d_out = d + (2.0f * cos_i) * nrm;
        } else if (M.type == GR_MAT_DIELECTRIC) {
          // chosen with u.x above; refraction by Snell's law in vector form
          const float e = 1.0f / n_rel;
          d_out = refracted ? e * d + (e * cos_i - cos_t) * nrm : d + (2.0f * cos_i) * nrm;
        } else {  // rough
          g_r = 2.0f * kw * M.sigma_h_um * cos_i;
          g_r *= g_r;
          float mreal;
          if (g_r > kGCont) {
            mreal = g_r;
          } else {
            float pm = expf(-g_r), cdf = pm;
            int mi = 0;
            while (u.x >= cdf && mi < 1000) {
              ++mi;
              pm *= g_r / (float)mi;
              cdf += pm;
            }
            const float eps = 4e-6f + 2e-7f * (float)mi;
            if (fabsf(u.x - cdf) < eps || (mi > 0 && fabsf(u.x - (cdf - pm)) < eps) || mi >= 1000) {
              atomicAdd(&p.ctr->ref_lobe, 1ull);
              mi = poisson_pick_fp64(bin_lambda_d(V, bin), M.sigma_h_um, cos_i, u.x);
            }
            mreal = (float)mi;
          }
          if (mreal == 0.0f) {
            d_out = d + (2.0f * cos_i) * nrm;
          } else {
            delta = 0;
            const float kl = kw * M.corr_len_um;
            const float sig = sqrtf(2.0f * mreal) / kl;
            float z0, z1;
            box_muller(u.y, u.z, z0, z1);
            float3 e1, e2;
            onb(nrm, e1, e2);
            const float3 dt = (sig * z0) * e1 + (sig * z1) * e2;
            const float3 to = t_mir + dt;
            const float tt = dot(to, to);
            if (tt >= 1.0f) {
              alive = false;
            } else {
              const float cz = sqrtf(1.0f - tt);
              d_out = to + cz * nrm;
              mis_rec = make_float4(dot(dt, dt), g_r, kl * kl, cz);
            }
          }
          if (HERO && alive) {
            // the class wavelengths' densities of the lobe term just
            // sampled (the cosine factor is common to all of them; g
            // scales with k^2 across the class): the specular term's
            // probability e^-g here; the m >= 1 density at the sampled
            // offset by k_density, on a compacted queue of such vertices
            // (here only a fraction of a warp's lanes would run the
            // series), from the lobe terms stored for MIS, the ratios and
            // the sample
            if (mreal == 0.0f) {
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                if (g == gh || hq[g] == 0.0f) continue;
                const float r = lambda * __frcp_rn(step_lambda(V, cstep, cls + g * Qv));
                const float gqg = g_r * (r * r);  // g at class wavelength g
                hq[g] *= gqg > kGCont ? 0.0f : expf(g_r - gqg);
              }
            } else {
              // (only a living companion's ratio needs the series)
#pragma unroll
              for (int g = 0; g < 4; ++g)
                if (g != gh && hq[g] != 0.0f) want_density = true;
            }
          }
        }
        if (HERO && M.type == GR_MAT_DIELECTRIC && M.cauchy_b_um2 != 0.0f) drop_companions();
        // --- next-event estimation toward an emitter (rough lobes only)
        if (WAVE && M.type == GR_MAT_ROUGH && (p.flags & GR_FLAG_NEE) && S.n_emitters > 0) {
          const float4 un = rng4(p.seed, V.view_index, pixel, smp, seg, kCallNeeDir);
          const int ne_cnt = S.n_emitters;
          int ei = (int)(un.x * (float)ne_cnt);
          if (ei > ne_cnt - 1) ei = ne_cnt - 1;
          const float3 nE = emitter_normal(S, ei);
          const gr_material EM = S.mats[S.emitters[ei].mat];
          const float kap = 1.0f / (s_ray2 + src_spread2(lambda, EM.coh_len_um));
          const float3 w = vmf_sample(-nE, kap, un.y, un.z);
          const float cos_o = dot(w, nrm);
          if (cos_o > 0.0f && g_r > 0.0f && emitter_reachable(S, ei, x, w)) {
            // the lobe density, the MIS weight and the measurement are
            // evaluated by k_shadow once the shadow ray reaches the emitter
            const float3 dtn = (w - dot(w, nrm) * nrm) - t_mir;
            const float kl = kw * M.corr_len_um;
            P.shd[slot] = make_float4(w.x, w.y, w.z, __int_as_float(ei | (seg << 16)));
            P.shc[slot] = make_float4(cn[0], NS == 4 ? cn[1] : 0.0f, NS == 4 ? cn[2] : 0.0f, NS == 4 ? cn[3] : 0.0f);
            P.shm[slot] = make_float4(dot(dtn, dtn), g_r, kl * kl, cos_o);
            if (ANISO) {
              // the vertex's footprint in the frame of the emitter direction
              const float3 xw = s_vector(nrm, -w, s_o);
              const AK Kw = ak_interaction(K, xyz(xfv), d, xw, w, nrm);
              P.nk0[slot] = make_float4(Kw.r11, Kw.r12, Kw.r22, Kw.i11);
              P.nk1[slot] = make_float4(Kw.i12, Kw.i22, 0.0f, 0.0f);
              P.nkf[slot] = make_float4(xw.x, xw.y, xw.z, 0.0f);
            }
            want_shadow = true;
          }
        }
        if (!WAVE) {
          // (x, beta2, rho) and the outgoing ray stay with the caller
          o = x;
          if (alive) {
            d = d_out;
            if (NS == 4) {
              const float3 xn = s_vector(nrm, -d_out, s_o);
              xfv = make_float4(xn.x, xn.y, xn.z, eta_next);
            } else {
              xfv.w = eta_next;
            }
          } else {
            done = true;
          }
        } else {
          // the vertex becomes the ray origin; (beta, rho) are unchanged by
          // the interaction (Eq. K_reflection_refraction, Eq. K_grating)
          P.od0[slot] = make_float4(x.x, x.y, x.z, beta2);
          if (alive) {
            P.od1[slot] = make_float4(d_out.x, d_out.y, d_out.z, rho);
            if (NS == 1) {
              P.tp[0][slot] = make_float4(T[0][0], eta_next, 0.0f, 0.0f);
            } else {
              for (int r = 0; r < 4; ++r) P.tp[r][slot] = make_float4(T[r][0], T[r][1], T[r][2], T[r][3]);
              const float3 xn = s_vector(nrm, -d_out, s_o);
              P.xf[slot] = make_float4(xn.x, xn.y, xn.z, eta_next);
            }
            if (!delta) P.mis[slot] = mis_rec;
            if (HERO) P.hq[slot] = make_float4(hq[0], hq[1], hq[2], hq[3]);
            if (ANISO) {
              // the footprint mapped onto the outgoing direction's frame
              const float3 xn = s_vector(nrm, -d_out, s_o);
              const AK Ko = ak_interaction(K, xyz(xfv), d, xn, d_out, nrm);
              P.ak0[slot] = make_float4(Ko.r11, Ko.r12, Ko.r22, Ko.i11);
              P.ak1[slot] = make_float4(Ko.i12, Ko.i22, 0.0f, 0.0f);
              if (NS == 1) P.xf[slot] = make_float4(xn.x, xn.y, xn.z, 0.0f);
            }
            P.meta[slot] = make_int4(m.x, m.y, meta_pack(kk, seg + 1, ST_ACTIVE, delta), hslot);
          } else {
            P.od1[slot] = make_float4(d.x, d.y, d.z, rho);
            P.meta[slot] = make_int4(m.x, m.y, meta_pack(kk, seg, ST_DONE, 0), hslot);
            // a pending next-event ray is measured in the next iteration:
            // the fold waits for it
            P.st8[slot] = want_shadow ? ST_WAIT : ST_DONE;
          }
        }
      }
    }
  }
