// tlbm_node.cuh -- one node's derivatives and collision, shared by the marching
// kernels of the pressure-tensor coupling (Semprebon, Krueger, Kusumaatmaja,
// arXiv:1511.02155), so that every kernel, tile and batch gives the same bits.
//
// These kernels are bound by instructions as much as by memory (FP16 D3Q19 issues
// in 62 % of all cycles, and FP64 has two lanes per SM and clock), so the node's
// arithmetic is written for few operations.  All products that feed a sum are
// explicit fused multiply-adds: the result does not depend on what the compiler
// contracts around the inlined call.
#pragma once

#include "tlbm_lattice.cuh"

namespace tlbm_dev {

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
// products that are added later: rounded here, never contracted into the sum
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }

// Derivatives of the three fields along one node's march, one plane at a time.
// The weights of the isotropic stencils (axis links twice, on D2Q9 four times,
// the diagonal ones) let each plane enter through a few sums of its in-plane
// neighbours: with da, db the differences across the node, s the sum of the axis
// neighbours, ea, eb, sd the same over the diagonal ones and t = W c + s
// (W = 2, on D2Q9 4),
//   12 d_a X = W da(m) + ea(m) + da(m-1) + da(m+1)      (d_b likewise)
//   12 d_m X = t(m+1) - t(m-1)
//    6 lap X = W s(m) + sd(m) + t(m-1) + t(m+1) - Z c(m),  Z = 24, on D2Q9 20.
// A plane's nine (three) ring values per field are read once instead of in three
// planes' stencils: 27 (9) reads and about 90 (30) operations a node in place of
// 57 (27) and 175 (80).
template <int Q, typename T>
struct Roll {
    static constexpr int D = Lat<Q>::D;
    static constexpr T W = D == 3 ? T(2) : T(4);
    T c[3], ua[3], ub[3], l[3], tm[3];  // centre plane: value and what its derivatives have so far
    T da[3], db[3], t[3];               // the newest plane's share in the next one

    // plane m+1 arrives: at(k, i, j) reads field k at in-plane offset (i, j),
    // c1 is the node's own value.  Returns the centre plane m's values: X, 12 grad
    // X in lattice axes and 6 lap X (meaningful from the third plane on).
    template <typename At>
    __device__ __forceinline__ void push(At at, const T (&c1)[3], T (&X)[3], T (&g12)[3][3], T (&l6)[3]) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T xp = at(k, 1, 0), xn = at(k, -1, 0);
            const T dan = xp - xn;
            T s = xp + xn, dbn = T(0), ea = T(0), eb = T(0), sd = T(0);
            if constexpr (D == 3) {
                const T yp = at(k, 0, 1), yn = at(k, 0, -1);
                dbn = yp - yn;
                s += yp + yn;
                const T pp = at(k, 1, 1), nn = at(k, -1, -1), pn = at(k, 1, -1), np = at(k, -1, 1);
                const T u = pp - nn, v = pn - np;
                ea = u + v;
                eb = u - v;
                sd = (pp + nn) + (pn + np);
            }
            const T tn = fma_(W, c1[k], s);
            // the centre plane is complete with this plane's share
            X[k] = c[k];
            g12[k][0] = ua[k] + dan;
            if constexpr (D == 3) {
                g12[k][1] = ub[k] + dbn;
                g12[k][2] = tn - tm[k];
            } else {
                g12[k][1] = tn - tm[k];
                g12[k][2] = T(0);
            }
            l6[k] = l[k] + tn;
            // this plane becomes the centre
            if constexpr (D == 3) {
                ua[k] = fma_(W, dan, ea) + da[k];
                ub[k] = fma_(W, dbn, eb) + db[k];
                l[k] = fma_(T(2), s, fma_(T(-24), c1[k], sd)) + t[k];
                db[k] = dbn;
            } else {
                ua[k] = fma_(W, dan, da[k]);
                l[k] = fma_(T(4), s, fma_(T(-20), c1[k], t[k]));
            }
            tm[k] = t[k];
            c[k] = c1[k];
            da[k] = dan;
            t[k] = tn;
        }
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < 3; ++k) c[k] = ua[k] = ub[k] = l[k] = tm[k] = da[k] = db[k] = t[k] = T(0);
    }
};

// Index of the gradient-term component of an edge link: the plane (a, b) it lies
// in as 0 xy, 1 yz, 2 zx, and the sign e_a e_b.
template <int Q>
__host__ __device__ constexpr int edge_plane(int i) {
    return Lat<Q>::cx(i) != 0 ? (Lat<Q>::cy(i) != 0 ? 0 : 2) : 1;
}
template <int Q>
__host__ __device__ constexpr int edge_sign(int i) {
    return edge_plane<Q>(i) == 0 ? Lat<Q>::cx(i) * Lat<Q>::cy(i)
                                 : (edge_plane<Q>(i) == 1 ? Lat<Q>::cy(i) * Lat<Q>::cz(i) : Lat<Q>::cz(i) * Lat<Q>::cx(i));
}

// Collision of one node and the store of its populations x* at node pointer out.
// fv, gv, kv: the pulled populations as stored (deviations from Fmt::bias); rd:
// their summed f (rho - 1 in the offset formats, else rho); X = (rho, phi, psi);
// j the momentum, g12, l6 the scaled derivatives of Roll (lattice axes).
// STREAM marks the stores evict-first.
//
// omega is folded into the equilibria, x* = (1 - omega) x + omega x_eq, and
// omega x_eq = EV +- OD for a pair of opposite links.  The gradient part needs
// G_ab = sum_XY K_XY d_a X d_b Y, which in the concentrations is the plain sum
// sum_m kappa_m d_a C_m d_b C_m; of its tensor weights only the trace, the link's
// own diagonal component and one off-diagonal one differ between links:
//   D3Q19 axis a: G_aa / 4 - tr / 9,   edge (a, b), normal c: G_cc / 24 - tr / 72 +- G_ab / 12
//   D2Q9  axis a: G_aa / 6 - tr / 18,  diagonal: -tr / 72 +- G_xy / 12
// so a link pair costs 17 operations for its six populations.
template <int Q, typename S, bool STREAM>
__device__ __forceinline__ void collide_node(unsigned char* out, const typename Store<S>::T (&fv)[Q],
                                             const typename Store<S>::T (&gv)[Q], const typename Store<S>::T (&kv)[Q],
                                             typename Store<S>::T rd, const typename Store<S>::T (&X)[3],
                                             const typename Store<S>::T (&j)[3],
                                             const typename Store<S>::T (&g12)[3][3],
                                             const typename Store<S>::T (&l6)[3], const Phys<typename Store<S>::T>& P) {
    using T = typename Store<S>::T;
    using F = Fmt<Q, S>;
    constexpr int D = Lat<Q>::D;
    constexpr bool OF = F::OFFSET;
    const T rho = X[0], phi = X[1], psi = X[2];
    const T inv = T(1) / rho;
    const T u[3] = {mul_(j[0], inv), mul_(j[1], inv), D == 3 ? mul_(j[2], inv) : T(0)};
    T uu = fma_(u[1], u[1], u[0] * u[0]);
    if constexpr (D == 3) uu = fma_(u[2], u[2], uu);
    const T huu = T(-1.5) * uu;

    // concentrations, their Laplacians and gradients (Sec. Auxiliary variables)
    const T C[3] = {T(0.5) * ((rho - psi) + phi), T(0.5) * ((rho - psi) - phi), psi};
    const T lC[3] = {T(0.5) * ((l6[0] - l6[2]) + l6[1]), T(0.5) * ((l6[0] - l6[2]) - l6[1]), l6[2]};
    // chemical potentials; pL = p_b - rho c_s^2 - alpha^2 sum_XY K_XY X lap Y, whose
    // last term is sum_m kappa_m C_m lap C_m in the concentrations
    T mu[3], pL = T(0);
    const T a6 = P.a2 * T(1.0 / 6.0);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const T c = C[m];
        const T b = fma_(-c, c, c);  // c (1 - c)
        const T al = a6 * lC[m];
        mu[m] = P.kappa[m] * fma_(b, fma_(T(-2), c, T(1)), -al);
        pL = fma_(P.kappa[m] * c, fma_(T(0.5) * b, fma_(T(-3), c, T(1)), -al), pL);
    }
    const T bf = fma_(rho, huu, fma_(T(3), pL, OF ? rd : rho));  // 3 p_b - ... (- 1 in the offset formats)
    const T mu_phi = T(0.5) * (mu[0] - mu[1]);
    const T mu_psi = fma_(T(-0.5), mu[0] + mu[1], mu[2]);
    const T bg = fma_(phi, huu, T(3) * P.gamma[0] * mu_phi);
    const T bk = fma_(psi, huu, T(3) * P.gamma[1] * mu_psi);

    // omega_f 3 alpha^2 G: diagonal Gd, off-diagonal Go (xy, yz, zx)
    T Gd[3] = {T(0), T(0), T(0)}, Go[3] = {T(0), T(0), T(0)};
    {
        const T sc = P.omega[0] * P.a2 * T(3.0 / 144.0);
        T gc[3][3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const T rp = g12[0][a] - g12[2][a];
            gc[0][a] = T(0.5) * (rp + g12[1][a]);
            gc[1][a] = T(0.5) * (rp - g12[1][a]);
            gc[2][a] = g12[2][a];
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const T k = sc * P.kappa[m];
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const T ka = k * gc[m][a];
                Gd[a] = fma_(ka, gc[m][a], Gd[a]);
                if (D == 3 || a == 0) Go[a] = fma_(ka, gc[m][(a + 1) % 3], Go[a]);
            }
        }
    }
    constexpr T wa = T(Lat<Q>::w(1)), we = T(Lat<Q>::w(Q - 1));  // axis and edge (diagonal) weights
    const T of = P.omega[0], og = P.omega[1], ok = P.omega[2];
    const T cf = T(1) - of, cg = T(1) - og, ck = T(1) - ok;
    const T tr = (Gd[0] + Gd[1]) + Gd[2];
    const T Bf = of * bf, Bg = og * bg, Bk = ok * bk;
    T fax[3], fed[3];  // f's even part without the velocity term: axis links, edges by plane
    if constexpr (D == 3) {
        const T ba = fma_(T(-1.0 / 9.0), tr, wa * Bf), be = fma_(T(-1.0 / 72.0), tr, we * Bf);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            fax[a] = fma_(T(0.25), Gd[a], ba);
            fed[a] = fma_(T(1.0 / 24.0), Gd[(a + 2) % 3], be);  // plane (a, a+1), normal a+2
        }
    } else {
        const T ba = fma_(T(-1.0 / 18.0), tr, wa * Bf);
        fax[0] = fma_(T(1.0 / 6.0), Gd[0], ba);
        fax[1] = fma_(T(1.0 / 6.0), Gd[1], ba);
        fax[2] = fed[1] = fed[2] = T(0);
        fed[0] = fma_(T(-1.0 / 72.0), tr, we * Bf);
    }
    const T of_r = of * rho, og_p = og * phi, ok_p = ok * psi;
    // odd parts: w times 3 omega X, not (3 w) times omega X: the rounded 1/3 and 1/12
    // are 3e-8 too large, the rounded w only 7e-9, and the momentum of every step
    // grows by that factor
    const T Of = T(3) * of_r, Og = T(3) * og_p, Ok = T(3) * ok_p;
    T sf = T(0), sg = T(0), sk = T(0);  // half sums of omega x_eq over the moving links (FP64)
    T qf = T(0), qg = T(0), qk = T(0);  // sums of the moving populations as stored
    T kn[Q];                            // packed: new k of directions whose word is not out yet
    auto put = [&](int s, int i, T d) {
        if (STREAM) F::st_stream_delta(out, s, i, d);
        else F::st_delta(out, s, i, d);
    };
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = opp<Q>(i);
        if (o < i) continue;
        const bool axis = i <= Lat<Q>::NAXIS;
        const T w = axis ? wa : we;
        T e = T(0), base;
        if (axis) {
            const int a = Lat<Q>::cx(i) ? 0 : (Lat<Q>::cy(i) ? 1 : 2);
            e = comp<Q>(i, a) > 0 ? u[a] : -u[a];
            base = fax[a];
        } else {
            const int p = edge_plane<Q>(i), b = (p + 1) % 3;
            const T x = comp<Q>(i, p) > 0 ? u[p] : -u[p];
            e = comp<Q>(i, b) > 0 ? x + u[b] : x - u[b];
            base = fma_(T(edge_sign<Q>(i) / 12.0), Go[p], fed[p]);
        }
        const T e2 = e * e;
        const T rw = T(4.5) * w;  // exact: 1/4, 1/2 and 1/8
        const T evf = fma_(rw * of_r, e2, base), of_w = w * Of;
        const T evg = fma_(rw * og_p, e2, w * Bg), og_w = w * Og;
        const T evk = fma_(rw * ok_p, e2, w * Bk), ok_w = w * Ok;
        if (!OF) {
            sf += evf;
            sg += evg;
            sk += evk;
        }
        const T v[6] = {fma_(cf, fv[i], fma_(of_w, e, evf)), fma_(cf, fv[o], fma_(-of_w, e, evf)),
                        fma_(cg, gv[i], fma_(og_w, e, evg)), fma_(cg, gv[o], fma_(-og_w, e, evg)),
                        fma_(ck, kv[i], fma_(ok_w, e, evk)), fma_(ck, kv[o], fma_(-ok_w, e, evk))};
        T q[4];  // the deviations as stored
        F::template st_fg_q<STREAM>(out, i, v[0], v[2], q[0], q[2]);
        F::template st_fg_q<STREAM>(out, o, v[1], v[3], q[1], q[3]);
        if (OF) {
            qf += q[0] + q[1];
            qg += q[2] + q[3];
        }
        if constexpr (F::PACKED) {
            // a k word goes out once both of its directions are collided
            kn[i] = v[4];
            kn[o] = v[5];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int d = h ? o : i, m = F::kmate(d), ml = m < opp<Q>(m) ? m : opp<Q>(m);
                if (ml > i || (ml == i && F::khalf(d) != 0)) continue;
                const int lo = F::khalf(d) == 0 ? d : m;
                T ql, qh;
                F::template st_kword_q<STREAM>(out, lo, kn[lo], kn[F::kmate(lo)], ql, qh);
                qk += ql + qh;
            }
        } else {
            F::template st_kk<STREAM>(out, i, v[4], v[5]);
            if (OF) qk += v[4] + v[5];
        }
    }
    if (OF) {
        // rest = moment - moving populations as stored (deviations for f): every
        // node keeps its rho, phi, psi through the rounding of the stored values
        put(0, 0, rd - qf);
        put(1, 0, phi - qg);
        put(2, 0, psi - qk);
    } else {
        // omega x_eq_0 = omega X - sum of omega x_eq over the moving links
        put(0, 0, fma_(cf, fv[0], fma_(T(-2), sf, of_r)));
        put(1, 0, fma_(cg, gv[0], fma_(T(-2), sg, og_p)));
        put(2, 0, fma_(ck, kv[0], fma_(T(-2), sk, ok_p)));
    }
}

}  // namespace tlbm_dev
