// tlbm_guo.cuh -- the forcing coupling of the ternary free-energy LB step: the
// alternative that Sec. Equations of Motion mentions beside the pressure-tensor
// equilibrium, in which the thermodynamic terms enter the momentum equation as
// a body force with the source of Guo, Zheng and Shi (2002).
//
// The force is the divergence of the non-ideal part of the paper's pressure
// tensor,
//   F_a = -d_b Pi_ab,   Pi_ab = P_ab - rho c_s^2 delta_ab,
//   Pi_ab = alpha^2 G_ab + delta_ab [p_b - rho c_s^2 - alpha^2 (tr G / 2 + L)],
//   G_ab = sum_XY K_XY d_a X d_b Y,   L = sum_XY K_XY X lap Y,
// which in the continuum equals -(rho grad mu_rho + phi grad mu_phi + psi grad
// mu_psi) and on a periodic lattice sums to zero exactly (total momentum is
// conserved).  f relaxes to the ideal-gas equilibrium (pressure rho c_s^2) at
// the fluid velocity u = (j + F/2) / rho and receives
//   S_i = (1 - omega_f / 2) w_i [3 (e_i - u).F + 9 (e_i.u)(e_i.F)];
// g and k keep the equilibria of Sec. The Lattice Boltzmann Equation at the
// same u.  Periodic lattices only.  The marching kernel k_guo_fused (below)
// does a step in one launch; the split step is three launches:
//   k_moments       rho, phi, psi of the pulled populations   -> mom[3][Np]
//   k_guo_pressure  Pi (3 components on D2Q9, 6 on D3Q19) and
//                   mu_phi, mu_psi of every node               -> aux[NA][Np]
//   k_guo_collide   pull, F from Pi at the neighbours, collide with the
//                   source, store x*(r) in the other buffer
#pragma once

#include "tlbm_kernels.cuh"
#include "tlbm_launch.cuh"

namespace tlbm_dev {

// layout of the forcing coupling's node arrays aux[NA][Np]
template <int Q>
struct GuoAux {
    static constexpr int D = Lat<Q>::D;
    // Pi components: xx yy xy (D2Q9); xx yy zz xy yz zx (D3Q19)
    static constexpr int NPI = D == 2 ? 3 : 6;
    static constexpr int MU = NPI;  // mu_phi at MU, mu_psi at MU + 1
    static constexpr int NA = NPI + 2;
    // first and second axis of component c
    __host__ __device__ static constexpr int ca(int c) { return c < D ? c : c - D; }
    __host__ __device__ static constexpr int cb(int c) { return c < D ? c : (D == 2 ? 1 : (c - 2) % 3); }
    // component of the axis pair (a, b)
    __host__ __device__ static constexpr int comp(int a, int b) {
        return a == b ? a : (D == 2 ? 2 : (a + b == 1 ? 3 : (a + b == 3 ? 4 : 5)));
    }
};

// Pi (GuoAux components) and mu_phi, mu_psi of one node from its fields X =
// (rho, phi, psi), their gradients grad[X][axis] and Laplacians lap[X].
template <int Q, typename T>
__device__ __forceinline__ void guo_node(const Phys<T>& P, const T (&X)[3], const T (&grad)[3][3],
                                         const T (&lap)[3], T (&pi)[GuoAux<Q>::NPI], T& mu_phi, T& mu_psi) {
    using A = GuoAux<Q>;
    // concentrations, chemical potentials and bulk pressure (Sec. Auxiliary
    // variables; p_b from the thermodynamic identity)
    const T C[3] = {(X[0] + X[1] - X[2]) * T(0.5), (X[0] - X[1] - X[2]) * T(0.5), X[2]};
    const T lC[3] = {(lap[0] + lap[1] - lap[2]) * T(0.5), (lap[0] - lap[1] - lap[2]) * T(0.5), lap[2]};
    T mu[3], pbx = T(0);  // pbx = p_b - rho c_s^2
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const T c = C[m], c1 = T(1) - c;
        mu[m] = P.kappa[m] * (c * c1 * (T(1) - T(2) * c) - P.a2 * lC[m]);
        pbx += P.kappa[m] * T(0.5) * c * c * c1 * (T(1) - T(3) * c);
    }
    // L = sum_XY K_XY X lap Y and G_ab = sum_XY K_XY d_a X d_b Y
    T Lp = T(0);
    T Kg[3][3];  // [X][b] = sum_Y K_XY d_b Y
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T s = T(0);
#pragma unroll
        for (int b = 0; b < 3; ++b) s += P.K[a][b] * lap[b];
        Lp += X[a] * s;
#pragma unroll
        for (int b = 0; b < 3; ++b)
            Kg[a][b] = P.K[a][0] * grad[0][b] + P.K[a][1] * grad[1][b] + P.K[a][2] * grad[2][b];
    }
    T G[A::NPI];
    T trG = T(0);
#pragma unroll
    for (int c = 0; c < A::NPI; ++c) {
        const int a = A::ca(c), b = A::cb(c);
        G[c] = grad[0][a] * Kg[0][b] + grad[1][a] * Kg[1][b] + grad[2][a] * Kg[2][b];
        if (a == b) trG += G[c];
    }
    const T iso = pbx - P.a2 * (T(0.5) * trG + Lp);
#pragma unroll
    for (int c = 0; c < A::NPI; ++c) pi[c] = P.a2 * G[c] + (A::ca(c) == A::cb(c) ? iso : T(0));
    mu_phi = (mu[0] - mu[1]) * T(0.5);
    mu_psi = mu[2] - (mu[0] + mu[1]) * T(0.5);
}

// The same from Roll's scaled derivatives (12 grad, 6 lap), in the concentrations:
// G_ab = sum_m kappa_m d_a C_m d_b C_m and L = sum_m kappa_m C_m lap C_m.
template <int Q, typename T>
__device__ __forceinline__ void guo_node12(const Phys<T>& P, const T (&X)[3], const T (&g12)[3][3], const T (&l6)[3],
                                           T (&pi)[GuoAux<Q>::NPI], T& mu_phi, T& mu_psi) {
    using A = GuoAux<Q>;
    const T C[3] = {T(0.5) * ((X[0] - X[2]) + X[1]), T(0.5) * ((X[0] - X[2]) - X[1]), X[2]};
    const T lC[3] = {T(0.5) * ((l6[0] - l6[2]) + l6[1]), T(0.5) * ((l6[0] - l6[2]) - l6[1]), l6[2]};
    T mu[3], pL = T(0), G[A::NPI];
    const T a6 = P.a2 * T(1.0 / 6.0), sc = P.a2 * T(1.0 / 144.0);
#pragma unroll
    for (int c = 0; c < A::NPI; ++c) G[c] = T(0);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const T c = C[m], b = fma_(-c, c, c), al = a6 * lC[m];
        mu[m] = P.kappa[m] * fma_(b, fma_(T(-2), c, T(1)), -al);
        pL = fma_(P.kappa[m] * c, fma_(T(0.5) * b, fma_(T(-3), c, T(1)), -al), pL);
        T gc[3];
#pragma unroll
        for (int a = 0; a < A::D; ++a) {
            const T rp = g12[0][a] - g12[2][a];
            gc[a] = m == 0 ? T(0.5) * (rp + g12[1][a]) : (m == 1 ? T(0.5) * (rp - g12[1][a]) : g12[2][a]);
        }
        const T km = sc * P.kappa[m];
#pragma unroll
        for (int q = 0; q < A::NPI; ++q) G[q] = fma_(km * gc[A::ca(q)], gc[A::cb(q)], G[q]);
    }
    T tr = T(0);
#pragma unroll
    for (int a = 0; a < A::D; ++a) tr += G[a];
    const T iso = fma_(T(-0.5), tr, pL);
#pragma unroll
    for (int q = 0; q < A::NPI; ++q) pi[q] = G[q] + (A::ca(q) == A::cb(q) ? iso : T(0));
    mu_phi = T(0.5) * (mu[0] - mu[1]);
    mu_psi = fma_(T(-0.5), mu[0] + mu[1], mu[2]);
}

// Pi and mu_phi, mu_psi of every node from the moment arrays (periodic).
template <int Q, typename T>
__global__ void __launch_bounds__(kThreads)
k_guo_pressure(Geom g, const T* __restrict__ mom, T* __restrict__ aux, Phys<T> P) {
    using A = GuoAux<Q>;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
         r += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        coords(g, r, x, y, z);
        T grad[3][3], lap[3];
        derivs<Q, T>(g, mom, x, y, z, r, grad, lap);
        const T X[3] = {mom[r], mom[g.Np + r], mom[2 * g.Np + r]};
        T pi[A::NPI], mp, ms;
        guo_node<Q, T>(P, X, grad, lap, pi, mp, ms);
#pragma unroll
        for (int c = 0; c < A::NPI; ++c) aux[c * g.Np + r] = pi[c];
        aux[A::MU * g.Np + r] = mp;
        aux[(A::MU + 1) * g.Np + r] = ms;
    }
}

// F = -div Pi at (x, y, z): F_a = -3 sum_i w_i sum_b e_ib Pi_ab(r + e_i).
template <int Q, typename T>
__device__ __forceinline__ void guo_force(const Geom& g, const T* __restrict__ aux, int x, int y, int z,
                                          T (&F)[3]) {
    using A = GuoAux<Q>;
    F[0] = F[1] = F[2] = T(0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const long long n = node(g, wrap(x + Lat<Q>::cx(i), g.nx), wrap(y + Lat<Q>::cy(i), g.ny),
                                 wrap(z + Lat<Q>::cz(i), g.nz));
        const int e[3] = {Lat<Q>::cx(i), Lat<Q>::cy(i), Lat<Q>::cz(i)};
        const T w = T(Lat<Q>::w(i));
#pragma unroll
        for (int a = 0; a < A::D; ++a) {
            T s = T(0);
#pragma unroll
            for (int b = 0; b < A::D; ++b)
                if (e[b]) s += T(e[b]) * aux[A::comp(a, b) * g.Np + n];
            F[a] -= w * s;
        }
    }
    F[0] *= T(3); F[1] *= T(3); F[2] *= T(3);
}

// Equilibria of direction i >= 1 under the forcing coupling, as deviations
// from Fmt::bias: f_eq = w_i rho (1 + 3 e.u + 4.5 (e.u)^2 - 1.5 u.u) (fb = rho,
// or rho - 1 where f is stored as f - w_i), g_eq = w_i (3 Gamma_phi mu_phi +
// phi (3 e.u + 4.5 (e.u)^2 - 1.5 u.u)), k_eq likewise with psi.
template <typename T>
struct GuoEq {
    T rho, phi, psi, fb, bg, bk, uu;
    __device__ __forceinline__ void eq(T w, T e, T& fe, T& ge, T& ke) const {
        const T q = T(3) * e + T(4.5) * e * e - T(1.5) * uu;
        fe = w * (fb + rho * q);
        ge = w * (bg + phi * q);
        ke = w * (bk + psi * q);
    }
};

// BGK of one node under the forcing coupling towards the equilibria plus the
// Guo source (f only), stored at node pointer cb.  f, gg, k: the pulled
// populations as stored (f as deviations where Fmt::OFFSET); rd their summed f
// (rho - 1 where OFFSET, else rho); j the momentum, F the force (lattice axes);
// bg, bk = 3 Gamma mu_phi, 3 Gamma mu_psi.  STREAM marks the stores evict-first.
// As in collide_node, omega is folded in and a pair of opposite links shares
//   EV = omega w (b + 9/2 rho e^2 - 3/2 rho u.u) + s w (9 e e.F - 3 u.F),
//   OD = w (3 omega rho e + 3 s e.F),  s = 1 - omega / 2, e = e_i.u (g, k: no F).
template <int Q, typename S, bool STREAM>
__device__ __forceinline__ void guo_collide_node(unsigned char* cb, const typename Store<S>::T (&f)[Q],
                                                 const typename Store<S>::T (&gg)[Q],
                                                 const typename Store<S>::T (&k)[Q], typename Store<S>::T rd,
                                                 const typename Store<S>::T (&j)[3], typename Store<S>::T phi,
                                                 typename Store<S>::T psi, const typename Store<S>::T (&F)[3],
                                                 typename Store<S>::T bg, typename Store<S>::T bk,
                                                 const Phys<typename Store<S>::T>& P) {
    using T = typename Store<S>::T;
    constexpr bool OF = Fmt<Q, S>::OFFSET;
    const T rho = OF ? T(1) + rd : rd;
    const T inv = T(1) / rho;
    const T u[3] = {mul_(fma_(T(0.5), F[0], j[0]), inv), mul_(fma_(T(0.5), F[1], j[1]), inv),
                    mul_(fma_(T(0.5), F[2], j[2]), inv)};
    const T uu = fma_(u[2], u[2], fma_(u[1], u[1], u[0] * u[0]));
    const T uF = fma_(u[2], F[2], fma_(u[1], F[1], u[0] * F[0]));
    const T of = P.omega[0], og = P.omega[1], ok = P.omega[2];
    const T cf = T(1) - of, cg = T(1) - og, ck = T(1) - ok, sc = fma_(T(-0.5), of, T(1));
    const T huu = T(-1.5) * uu;
    const T Bf = of * fma_(rho, huu, OF ? rd : rho), Bg = og * fma_(phi, huu, bg), Bk = ok * fma_(psi, huu, bk);
    const T Rf = of * rho, Rg = og * phi, Rk = ok * psi;
    const T Of = T(3) * Rf, Og = T(3) * Rg, Ok = T(3) * Rk;
    const T s3 = T(3) * sc, s9 = T(9) * sc, S0 = T(-3) * sc * uF;
    T sf = T(0), sg = T(0), sk = T(0);  // half sums of omega x_eq over the moving links (FP64)
    T qf = T(0), qg = T(0), qk = T(0);  // sums of the moving populations as stored
    auto put = [&](int s, T d) {
        if (STREAM) Fmt<Q, S>::st_stream_delta(cb, s, 0, d);
        else Fmt<Q, S>::st_delta(cb, s, 0, d);
    };
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = opp<Q>(i);
        if (o < i) continue;
        const T w = T(Lat<Q>::w(i)), rw = T(4.5) * w;
        T e = T(0), eF = T(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int c = comp<Q>(i, a);
            if (c > 0) e += u[a], eF += F[a];
            if (c < 0) e -= u[a], eF -= F[a];
        }
        const T e2 = e * e;
        const T qvf = fma_(rw * Rf, e2, w * Bf);
        const T evf = fma_(w, fma_(s9 * e, eF, S0), qvf), odf = mul_(w, fma_(Of, e, s3 * eF));
        const T evg = fma_(rw * Rg, e2, w * Bg), odg = w * Og;
        const T evk = fma_(rw * Rk, e2, w * Bk), odk = w * Ok;
        if (!OF) {
            sf += qvf;
            sg += evg;
            sk += evk;
        }
        const T v[6] = {fma_(cf, f[i], evf + odf), fma_(cf, f[o], evf - odf),
                        fma_(cg, gg[i], fma_(odg, e, evg)), fma_(cg, gg[o], fma_(-odg, e, evg)),
                        fma_(ck, k[i], fma_(odk, e, evk)), fma_(ck, k[o], fma_(-odk, e, evk))};
        if (OF) {
            qf += Fmt<Q, S>::qdelta_d(i, v[0]) + Fmt<Q, S>::qdelta_d(o, v[1]);
            qg += Fmt<Q, S>::qdelta_d(i, v[2]) + Fmt<Q, S>::qdelta_d(o, v[3]);
            qk += Fmt<Q, S>::qdelta_d(i, v[4]) + Fmt<Q, S>::qdelta_d(o, v[5]);
        }
        Fmt<Q, S>::template st_fg<STREAM>(cb, i, v[0], v[2]);
        Fmt<Q, S>::template st_fg<STREAM>(cb, o, v[1], v[3]);
        Fmt<Q, S>::template st_kk<STREAM>(cb, i, v[4], v[5]);
    }
    if (OF) {
        // the source sums to zero over i: the rest population is what keeps
        // the node's rho, phi, psi through the storage rounding
        put(0, rd - qf);
        put(1, phi - qg);
        put(2, psi - qk);
    } else {
        put(0, fma_(T(Lat<Q>::w(0)), S0, fma_(cf, f[0], fma_(T(-2), sf, Rf))));
        put(1, fma_(cg, gg[0], fma_(T(-2), sg, Rg)));
        put(2, fma_(ck, k[0], fma_(T(-2), sk, Rk)));
    }
}

// Collide and stream every node of a periodic lattice under the forcing
// coupling: pull, moments, F from Pi at the neighbours, guo_collide_node.
template <int Q, typename S>
__global__ void __launch_bounds__(kThreads)
k_guo_collide(Geom g, const S* __restrict__ src, S* __restrict__ dst,
              const typename Store<S>::T* __restrict__ aux, Phys<typename Store<S>::T> P) {
    using T = typename Store<S>::T;
    using A = GuoAux<Q>;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
         r += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        coords(g, r, x, y, z);
        unsigned char* cb = reinterpret_cast<unsigned char*>(dst) + node_off<Q, S>(g, x, y, z);
        T f[Q], gg[Q], k[Q];  // f as stored (deviation where OFFSET), g and k as they are
        T rd = T(0), j[3] = {T(0), T(0), T(0)}, phi = T(0), psi = T(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            f[i] = pull_delta<Q, S, false>(g, src, nullptr, 0, i, x, y, z);
            gg[i] = pull_delta<Q, S, false>(g, src, nullptr, 1, i, x, y, z);
            k[i] = pull_delta<Q, S, false>(g, src, nullptr, 2, i, x, y, z);
            rd += f[i];
            if (Lat<Q>::cx(i)) j[0] += T(Lat<Q>::cx(i)) * f[i];
            if (Lat<Q>::cy(i)) j[1] += T(Lat<Q>::cy(i)) * f[i];
            if (Lat<Q>::cz(i)) j[2] += T(Lat<Q>::cz(i)) * f[i];
            phi += gg[i];
            psi += k[i];
        }
        T F[3];
        guo_force<Q, T>(g, aux, x, y, z, F);
        guo_collide_node<Q, S, false>(cb, f, gg, k, rd, j, phi, psi, F, T(3) * P.gamma[0] * aux[A::MU * g.Np + r],
                               T(3) * P.gamma[1] * aux[(A::MU + 1) * g.Np + r], P);
    }
}

// Populations at the forcing coupling's equilibrium of the fields in mom (with
// mu_phi, mu_psi in aux; stored momentum rho u, u[3][N] or NULL for rest),
// scattered so that the pull yields x_i(r) = x_eq_i(r).  Periodic lattices.
template <int Q, typename S>
__global__ void __launch_bounds__(kThreads)
k_guo_init(Geom g, S* __restrict__ dst, const typename Store<S>::T* __restrict__ mom,
           const typename Store<S>::T* __restrict__ aux, const double* __restrict__ u,
           Phys<typename Store<S>::T> P) {
    using T = typename Store<S>::T;
    using A = GuoAux<Q>;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
         r += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        coords(g, r, x, y, z);
        GuoEq<T> E;
        E.rho = mom[r]; E.phi = mom[g.Np + r]; E.psi = mom[2 * g.Np + r];
        E.fb = E.rho;
        const T v[3] = {u ? T(u[r]) : T(0), u ? T(u[g.N + r]) : T(0), u ? T(u[2 * g.N + r]) : T(0)};
        E.uu = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        E.bg = T(3) * P.gamma[0] * aux[A::MU * g.Np + r];
        E.bk = T(3) * P.gamma[1] * aux[(A::MU + 1) * g.Np + r];
        T eqv[3][Q];
        T sf = T(0), sg = T(0), sk = T(0);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            T e = T(0);
            if (Lat<Q>::cx(i)) e += T(Lat<Q>::cx(i)) * v[0];
            if (Lat<Q>::cy(i)) e += T(Lat<Q>::cy(i)) * v[1];
            if (Lat<Q>::cz(i)) e += T(Lat<Q>::cz(i)) * v[2];
            E.eq(T(Lat<Q>::w(i)), e, eqv[0][i], eqv[1][i], eqv[2][i]);
            sf += eqv[0][i]; sg += eqv[1][i]; sk += eqv[2][i];
        }
        eqv[0][0] = E.rho - sf; eqv[1][0] = E.phi - sg; eqv[2][0] = E.psi - sk;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int xs = wrap(x - Lat<Q>::cx(i), g.nx), ys = wrap(y - Lat<Q>::cy(i), g.ny),
                      zs = wrap(z - Lat<Q>::cz(i), g.nz);
#pragma unroll
            for (int s = 0; s < 3; ++s) pst<Q, S>(dst, g, s, i, xs, ys, zs, eqv[s][i]);
        }
    }
}

// Fluid velocity under the forcing coupling: u (holding j / rho) += F / (2 rho),
// with rho from mom and F from Pi in aux.  Periodic lattices.
template <int Q, typename T>
__global__ void __launch_bounds__(kThreads)
k_guo_velocity(Geom g, const T* __restrict__ mom, const T* __restrict__ aux, double* __restrict__ u) {
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
         r += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        coords(g, r, x, y, z);
        T F[3];
        guo_force<Q, T>(g, aux, x, y, z, F);
        const double h = 0.5 / (double)mom[r];
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a * g.N + r] += h * (double)F[a];
    }
}

// ------------------------------------------------ one marching kernel per step

// The forcing coupling's step as one kernel (periodic lattices), on the
// marching scheme of k_fused: a block owns a TX x TY column tile and marches a
// chunk of planes.  F at r needs Pi at r's neighbours, and Pi the derivatives
// of the moments, so the block keeps a two-node halo of moments and a one-node
// halo of Pi and works two planes ahead:
//   M(m+2): moments of plane m+2 over tile + two-node halo   -> moment ring
//   barrier
//   P(m+1): Pi of plane m+1 over tile + one-node halo          -> Pi ring,
//           mu_phi, mu_psi of the tile                         -> mu ring
//   barrier
//   C(m):   F from the Pi ring, pull, guo_collide_node, store x*(r).
// Ring slots: moments five (a fast warp writes plane m+2 while a slow one still
// reads planes m-2..m in C(m-1)); Pi three (P(m+1) starts after the barrier
// that every warp reaches only once its C(m-1), the last reader of plane
// m-2, is done); momentum and mu four.
// What it costs is the halo: with 32x4 tiles on D3Q19 the moments of 288 nodes and Pi
// of 204 for 128 of the tile.  Tiles of 32x8 (432 and 340 for 256), mu kept from P
// instead of a second set of derivatives in C, and link pairs in the collision:
// 128^3 FP32 351 us a step before, 345 after (338 with totals in pairs of floats, which
// hold fewer bits).
template <int Q, typename S>
constexpr int guo_smem(int TX, int TY) {
    const int b = Q == 19 ? 1 : 0, hn = (TX + 4) * (TY + 4 * b), pn = (TX + 2) * (TY + 2 * b);
    return (int)sizeof(typename Store<S>::T) * (15 * hn + 3 * GuoAux<Q>::NPI * pn + 24 * TX * TY);
}

template <int Q, typename S, int TX, int TY>
__device__ __forceinline__ void guo_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                         const Phys<typename Store<S>::T>& P, double* __restrict__ partials,
                                         const int bid) {
    extern __shared__ __align__(16) unsigned char tlbm_smem[];
    using T = typename Store<S>::T;
    using A = Axes<Q>;
    using GA = GuoAux<Q>;
    constexpr int D = Lat<Q>::D;
    constexpr int H = 2;                  // moment halo along a
    constexpr int HB = (D == 3) ? 2 : 0;  // moment halo along b
    constexpr int HW = TX + 2 * H;
    constexpr int HH = TY + 2 * HB;
    constexpr int HN = HW * HH;
    constexpr int NT = TX * TY;
    constexpr int KS = (HN + NT - 1) / NT;  // moment-region nodes per thread
    constexpr int PB = (D == 3) ? 1 : 0;    // Pi halo along b (one node along a)
    constexpr int PW = TX + 2;
    constexpr int PN = PW * (TY + 2 * PB);
    constexpr int KP = (PN + NT - 1) / NT;  // Pi-region nodes per thread
    constexpr int NPI = GA::NPI;
    static_assert(D == 3 || TY == 1, "2-D tiles are one row");
    static_assert(KS <= 3 && KP <= 2, "region nodes per thread");

    // dynamic shared memory (guo_smem)
    T (*const sm)[3][HN] = reinterpret_cast<T(*)[3][HN]>(tlbm_smem);  // rho, phi, psi over tile + two-node halo
    T (*const sp)[NPI][PN] = reinterpret_cast<T(*)[NPI][PN]>(tlbm_smem + sizeof(T) * 15 * HN);  // Pi, tile + one node
    // j (marching axes), summed f, mu_phi, mu_psi of the tile
    T (*const sj)[6][NT] = reinterpret_cast<T(*)[6][NT]>(tlbm_smem + sizeof(T) * (15 * HN + 3 * NPI * PN));

    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int tileA = bid % g.tilesA;
    const int rest = bid / g.tilesA;
    const int tileB = rest % g.tilesB;
    const int chunk = rest / g.tilesB;
    const int A0 = tileA * TX, B0 = tileB * TY;
    const int M0 = (int)((long long)chunk * g.NM / g.NC);
    const int M1 = (int)((long long)(chunk + 1) * g.NM / g.NC);
    const bool active = (A0 + tx < g.NA) && (B0 + ty < g.NB);

    // moment-region nodes of this thread: pull-source byte offsets along a, rows along b
    int xc[KS][3], yb[KS][3];
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const int h = min(tid + k * NT, HN - 1);
        const int aa = modp(A0 + h % HW - H, g.NA);
        const int bb = (D == 3) ? modp(B0 + h / HW - HB, g.NB) : 0;
        const int xs[3] = {wrap1(aa - 1, g.NA), aa, wrap1(aa + 1, g.NA)};
#pragma unroll
        for (int c = 0; c < 3; ++c) xc[k][c] = (xs[c] >> 5) * (int)Fmt<Q, S>::CHUNK + (xs[c] & 31) * Fmt<Q, S>::ESZ;
        yb[k][0] = (D == 3) ? wrap1(bb - 1, g.NB) : 0;
        yb[k][1] = bb;
        yb[k][2] = (D == 3) ? wrap1(bb + 1, g.NB) : 0;
    }
    const unsigned char* srcb = reinterpret_cast<const unsigned char*>(src);

    // M: moments of plane m over the two-node halo region
    auto moments_plane = [&](int m) {
        const int mm = modp(m, g.NM), slot = modp(m, 5), js = modp(m, 4);
        const int zr[3] = {wrap1(mm - 1, g.NM), mm, wrap1(mm + 1, g.NM)};
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int h = tid + k * NT;
            if (h >= HN) break;
            T rd = T(0), ja = T(0), jb = T(0), jm = T(0), phi = T(0), psi = T(0);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const unsigned char* p =
                    srcb + ((long long)zr[1 - A::cm(i)] * g.NB + yb[k][1 - A::cb(i)]) * g.rowstride + xc[k][1 - A::ca(i)];
                T f, gp;
                if (Fmt<Q, S>::PAIRED && i > 0) Fmt<Q, S>::ld_fg(p, i, f, gp);  // one lane word
                else f = Fmt<Q, S>::ld_delta(p, 0, i), gp = Fmt<Q, S>::ld_delta(p, 1, i);
                rd += f;
                if (A::ca(i)) ja += T(A::ca(i)) * f;
                if (A::cb(i)) jb += T(A::cb(i)) * f;
                if (A::cm(i)) jm += T(A::cm(i)) * f;
                phi += gp;
                psi += Fmt<Q, S>::ld_delta(p, 2, i);
            }
            sm[slot][0][h] = Fmt<Q, S>::OFFSET ? T(1) + rd : rd;
            sm[slot][1][h] = phi;
            sm[slot][2][h] = psi;
            const int hx = h % HW, hy = h / HW;
            if (hx >= H && hx < H + TX && hy >= HB && hy < HB + TY) {
                const int t = (hy - HB) * TX + (hx - H);
                sj[js][0][t] = ja;
                sj[js][1][t] = jb;
                sj[js][2][t] = jm;
                sj[js][3][t] = rd;
            }
        }
    };

    // P: Pi of plane q over the one-node halo region, mu of the tile
    auto pi_plane = [&](int q) {
        const int slot = modp(q, 3), js = modp(q, 4);
        const int s0 = modp(q - 1, 5), s1 = modp(q, 5), s2 = modp(q + 1, 5);
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const int pn = tid + k * NT;
            if (pn >= PN) break;
            const int py = pn / PW, px = pn % PW;
            const int h = (py + HB - PB) * HW + px + H - 1;  // the same node in the moment region
            T X[3], g12[3][3], l6[3], pi[NPI], mp, ms;
            Roll<Q, T> roll;
            roll.clear();
            auto push = [&](int sl) {
                const T c1[3] = {sm[sl][0][h], sm[sl][1][h], sm[sl][2][h]};
                roll.push([&](int c, int i, int jj) -> T { return sm[sl][c][h + jj * HW + i]; }, c1, X, g12, l6);
            };
            push(s0);
            push(s1);
            push(s2);
            guo_node12<Q, T>(P, X, g12, l6, pi, mp, ms);
#pragma unroll
            for (int c = 0; c < NPI; ++c) sp[slot][c][pn] = pi[c];
            if (px >= 1 && px <= TX && py >= PB && py < PB + TY) {
                const int t = (py - PB) * TX + px - 1;
                sj[js][4][t] = mp;
                sj[js][5][t] = ms;
            }
        }
    };

    constexpr bool PAIR = Fmt<Q, S>::OFFSET && !(Q == 19 && sizeof(S) == 4);
    MassSum<T, PAIR> msum;

    grid_ready();
    moments_plane(M0 - 2);
    moments_plane(M0 - 1);
    moments_plane(M0);
    moments_plane(M0 + 1);
    __syncthreads();
    pi_plane(M0 - 1);
    pi_plane(M0);
    __syncthreads();

    const int c0 = (ty + HB) * HW + tx + H;   // this thread's tile node in the moment region
    const int p0 = (ty + PB) * PW + tx + 1;   // ... and in the Pi region
    // the thread's own node: byte offsets of a-1, a, a+1 and rows b-1, b, b+1
    int xo[3], yo[3];
    {
        const int aa = modp(A0 + tx, g.NA), bb = (D == 3) ? modp(B0 + ty, g.NB) : 0;
        const int xs[3] = {wrap1(aa - 1, g.NA), aa, wrap1(aa + 1, g.NA)};
#pragma unroll
        for (int c = 0; c < 3; ++c) xo[c] = (xs[c] >> 5) * (int)Fmt<Q, S>::CHUNK + (xs[c] & 31) * Fmt<Q, S>::ESZ;
        yo[0] = (D == 3) ? wrap1(bb - 1, g.NB) : 0;
        yo[1] = bb;
        yo[2] = (D == 3) ? wrap1(bb + 1, g.NB) : 0;
    }
    for (int m = M0; m < M1; ++m) {
        moments_plane(m + 2);
        __syncthreads();
        pi_plane(m + 1);
        __syncthreads();
        if (!active) continue;

        const int s0 = modp(m, 5);
        const T X0[3] = {sm[s0][0][c0], sm[s0][1][c0], sm[s0][2][c0]};
        // F_a = -3 sum_i w_i sum_b e_ib Pi_ab(r + e_i) (lattice axes)
        T F[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const int sl = modp(m + A::cm(i), 3);
            const int pn = p0 + A::cb(i) * PW + A::ca(i);
            const int e[3] = {Lat<Q>::cx(i), Lat<Q>::cy(i), Lat<Q>::cz(i)};
            const T w = T(Lat<Q>::w(i));
#pragma unroll
            for (int a = 0; a < D; ++a) {
                T sacc = T(0);
#pragma unroll
                for (int b = 0; b < D; ++b)
                    if (e[b]) sacc += T(e[b]) * sp[sl][GA::comp(a, b)][pn];
                F[a] -= w * sacc;
            }
        }
        F[0] *= T(3); F[1] *= T(3); F[2] *= T(3);
        const int t = ty * TX + tx, js = modp(m, 4);
        const T rdc = sj[js][3][t];
        const T jl[3] = {sj[js][0][t], D == 3 ? sj[js][1][t] : sj[js][2][t], D == 3 ? sj[js][2][t] : T(0)};
        if constexpr (PAIR) msum.add(rdc, X0[1], X0[2]);
        else msum.add(rho_total<Q, S>(rdc), X0[1], X0[2]);

        // pulled populations of the node at plane m (deviations where OFFSET), their
        // last use: evict-first for FP32, as in the solid-aware kernel
        constexpr bool HL = sizeof(S) == 4;
        const int zr[3] = {wrap1(m - 1, g.NM), m, wrap1(m + 1, g.NM)};
        T fv[Q], gv[Q], kv[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const unsigned char* p =
                srcb + ((long long)zr[1 - A::cm(i)] * g.NB + yo[1 - A::cb(i)]) * g.rowstride + xo[1 - A::ca(i)];
            if (Fmt<Q, S>::PAIRED && i > 0) {
                Fmt<Q, S>::template ld_fg<HL>(p, i, fv[i], gv[i]);
            } else {
                fv[i] = HL ? Fmt<Q, S>::ld_last_delta(p, 0, i) : Fmt<Q, S>::ld_delta(p, 0, i);
                gv[i] = HL ? Fmt<Q, S>::ld_last_delta(p, 1, i) : Fmt<Q, S>::ld_delta(p, 1, i);
            }
            kv[i] = HL ? Fmt<Q, S>::ld_last_delta(p, 2, i) : Fmt<Q, S>::ld_delta(p, 2, i);
        }
        unsigned char* out =
            reinterpret_cast<unsigned char*>(dst) + ((long long)m * g.NB + yo[1]) * g.rowstride + xo[1];
        guo_collide_node<Q, S, HL>(out, fv, gv, kv, rdc, jl, X0[1], X0[2], F, T(3) * P.gamma[0] * sj[js][4][t],
                                   T(3) * P.gamma[1] * sj[js][5][t], P);
    }
    double mr, mp, ms;
    msum.get(mr, mp, ms);
    block_sum3(mr, mp, ms);
    if (tid == 0) put_block_sums(g, partials, bid, mr, mp, ms);
}

template <int Q, typename S, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, 512 / (TX * TY))
k_guo_fused(MGeom g, const S* __restrict__ src, S* __restrict__ dst, Phys<typename Store<S>::T> P,
            double* __restrict__ partials) {
    guo_body<Q, S, TX, TY>(g, src, dst, P, partials, blockIdx.x);
}

// One step of the forcing coupling with the marching kernel (tile from fused_cfg).
template <int Q, typename S>
inline cudaError_t guo_fused_step(tlbm_host::DevState& d, const Phys<typename Store<S>::T>& P, cudaStream_t st) {
    const FusedCfg<Q> c = fused_cfg<Q>(d);
    const MGeom g = mgeom<Q, S>(d, c);
    const long long nb = (long long)g.tilesA * g.tilesB * g.NC;
    if (nb > 0x7fffffffLL || nb > d.partials_cap) return cudaErrorInvalidConfiguration;
    const S* src = static_cast<const S*>(d.pop[d.cur]);
    S* dst = static_cast<S*>(d.pop[1 - d.cur]);
    cudaError_t e;
    if constexpr (Q == 19) {
        constexpr int TX = sizeof(S) == 8 ? 16 : 32, TY = sizeof(S) == 8 ? 4 : 8;
        e = launch_smem(k_guo_fused<Q, S, TX, TY>, guo_smem<Q, S>(TX, TY), TX * TY, 512 / (TX * TY), nb, st, g, src, dst, P,
                        d.partials);
    } else {
        e = launch_smem(k_guo_fused<Q, S, 128, 1>, guo_smem<Q, S>(128, 1), 128, 4, nb, st, g, src, dst, P, d.partials);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace tlbm_dev
