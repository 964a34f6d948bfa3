// tlbm_launch.cuh -- host side of the marching kernels: tiles, chunks, launches and
// batches.
#pragma once

#include <vector>

#include "tlbm_bulk.cuh"
#include "tlbm_fused.cuh"

namespace tlbm_dev {

// ------------------------------------------------------------ host side

// grid of a grid-stride kernel of 256 threads over n items: at most 8 blocks
// per SM (results do not depend on it)
inline int grid_of(long long n, int sms) {
    const long long b = (n + 255) / 256, cap = 8LL * (sms < 1 ? 1 : sms);
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// Cost of marching nb blocks of mc planes each, up to a factor.  A block pays for
// its planes plus halo prologue planes; a plane of one of b blocks that share an
// SM (res fit) takes 0.25 + 0.19 b' times a full SM's plane, b' = 4 b / res: alone
// a block waits out the latency of its loads, together they fill each other's
// waits.  Blocks beyond what fits wait for whole rounds; over many rounds the
// blocks drift apart and only the sum counts.  FP64 is bound by its few FP64
// units: there every node's operations count, about 400 for a collision and 72
// for the moments of a (node, halo) pair, and two blocks hide each other.
// Against the measured times of 14 lattices (64^2 .. 1000x701, 40^3 .. 160^2x96)
// over chunks of 1 .. 64 planes the cheapest chunk of this model is within 8 % of
// the fastest measured; halving 64 or 16 until 4 blocks per SM are reached, the
// earlier rule, lost up to 27 % (FP32, one step: 64x64 15.4 us against 11.3,
// 96^3 117.4 against 102.9, walled 144x128x80 299 against 267).
inline double march_cost(double nb, int mc, int halo, int res, int sms, bool dbl) {
    const double full = (double)res * sms;
    if (dbl) {
        const double per = nb / sms, b = per > 8.0 ? per : (double)(long long)(per + 0.9999);
        return (mc * 400.0 + (mc + halo) * 72.0) * (b < 2.0 ? 1.3 : b);
    }
    auto plane = [&](double b) { return 0.25 + 0.19 * 4.0 * b / res; };
    const double rounds = nb / full;
    if (rounds >= 4.0) return (mc + halo) * plane(res) * rounds;
    const double whole = (double)(long long)rounds;
    const double rest = nb - whole * full;
    const double b = (double)(long long)((rest + sms - 1) / sms);
    return (mc + halo) * (whole * plane(res) + (rest > 0 ? plane(b) : 0.0));
}

// Planes per block (chunk) of one marching launch over n lattices with cols[k]
// tile columns of nm[k] planes: the cheapest by march_cost whose block sums fit
// (caps[k]).  At most 64 planes in 2-D; in 3-D 16 once the grid fills the device
// eight times over (256^3 FP32: 16 planes 0.692 of HBM, 24..128 planes 0.66..0.69:
// blocks that start together share their halo rows in L2).
inline int pick_chunk(const long long* cols, const int* nm, const long long* caps, int n, int halo, int res, int sms,
                      bool three_d, bool dbl) {
    double best = 0.0;
    int bmc = 0;
    for (int mc = three_d ? 2 : 1; mc <= 64; ++mc) {
        double nb = 0.0;
        int used = 0;
        bool fits = true;
        for (int k = 0; k < n; ++k) {
            const int nc = (nm[k] + mc - 1) / mc, per = (nm[k] + nc - 1) / nc;
            nb += (double)cols[k] * nc;
            used = per > used ? per : used;
            fits = fits && cols[k] * nc <= caps[k];
        }
        if (!fits) continue;
        const double c = march_cost(nb, used, halo, res, sms, dbl);
        if (three_d && used > 16 && nb >= 8.0 * res * sms) continue;
        if (bmc == 0 || c < best) {
            best = c;
            bmc = mc;
        }
    }
    return bmc == 0 ? 64 : bmc;
}

template <int Q>
struct FusedCfg {
    int TX, TY, MC;
    int mode;
    int shape;  // D2Q9 shape
    // prologue planes a block recomputes, and blocks per SM (blocks_per_sm)
    int halo(const tlbm_host::DevState& d) const { return d.solid || d.coupling ? 4 : 2; }
    int res(const tlbm_host::DevState& d) const {
        if (Q == 19 && d.prec != 0 && !d.solid && !d.coupling) return d.prec == 1 ? BulkShape<float>::BPS : BulkShape<__half>::BPS;  // k_bulk
        return d.prec == 0 && TX == 32 ? 8 : 512 / (TX * TY);
    }
};

// d.tile = shape | mode << 4 | chunk << 8: shape 0 = default.  D3Q19 has one
// kernel per storage format (FP32 and 16-bit: k_bulk; double: k_fused, 16x8 nodes);
// its shapes are accepted and change nothing.  D2Q9 shape 0 = 5: 128-node rows with
// all 27 values staged, 1 = 128, 2 = 256, 3 = 64, 4 = 128 with the 18 lane-shifted
// values staged.  mode (shapes 1..3) bit 0: interleaved border loads; bit 1: early
// phase-C loads; bit 2: per-warp L2 prefetch three planes ahead; 8 / 9: evict-first
// stores / stores and collision loads (12, 13 with the prefetch).  mode 0 is the
// default for the shape (13); 6 selects the plain loop.  chunk = planes per block
// (0 = pick_chunk).
// D2Q9 in double: rows of 32 nodes (one warp) where rows of 128 in chunks of four
// planes leave SMs idle; wider rows recompute fewer halo moments.
// A batch launches one tile for all members: narrow only if every member is.
inline bool narrow_rows(const tlbm_host::DevState& d) { return !d.rows128 && d.N < 512LL * d.sms; }


template <int Q>
inline FusedCfg<Q> fused_cfg(const tlbm_host::DevState& d) {
    const bool dbl = d.prec == 0;  // double storage: one default shape only
    const int tile = d.checked ? 0 : d.tile;  // the checked kernels use the default tile
    const int variant = dbl ? 0 : (tile & 15);
    int mc = tile >> 8;
    FusedCfg<Q> c{};
    if (d.coupling) {
        // forcing coupling (k_guo_fused): the solid-aware kernel's tiles (two-node halo)
        c.TX = Q == 19 ? (dbl ? 16 : 32) : 128;
        c.TY = Q == 19 ? 4 : 1;
    } else if (d.solid) {
        // solid-aware kernel: a fixed tile per lattice (D3Q19 in double: 16x4 keeps
        // its five-plane rings under the 48 KB static shared-memory limit)
        c.TX = Q == 19 ? (dbl ? 16 : 32)
                       : (dbl ? (narrow_rows(d) ? 32 : 128) : (variant == 2 ? 256 : (variant == 3 ? 64 : 128)));
        c.TY = Q == 19 ? 4 : 1;
    } else if (Q == 19 && dbl) {
        c.TX = 16;  // double storage: a smaller tile keeps the static shared ring small
        c.TY = 8;
    } else if (Q == 19) {
        c.TX = 32;  // k_bulk
        c.TY = 4;
    } else {
        const int v = variant == 0 ? 5 : variant;  // 128-node rows with staging measured fastest
        c.TX = dbl ? (narrow_rows(d) ? 32 : 128) : (v == 2 ? 256 : (v == 3 ? 64 : 128));
        c.TY = 1;
        c.shape = v;
    }
    c.mode = dbl ? 0 : ((tile >> 4) & 15);
    if (c.mode == 0) c.mode = 13;  // D2Q9: prefetch, evict-first stores and collision loads
    const int NA = d.nx;
    const int NB = (Q == 19) ? d.ny : 1;
    const int NM = (Q == 19) ? d.nz : d.ny;
    if (mc <= 0) {
        const long long cols = (long long)((NA + c.TX - 1) / c.TX) * ((NB + c.TY - 1) / c.TY);
        mc = pick_chunk(&cols, &NM, &d.partials_cap, 1, c.halo(d), c.res(d), d.sms, Q == 19, dbl);
    }
    c.MC = mc < 1 ? 1 : (mc > NM ? NM : mc);
    return c;
}

template <int Q, typename S>
inline bool fused_supported(const tlbm_host::DevState& d) {
    return d.solid == nullptr || d.nbm != nullptr;
}

template <int Q, typename S>
inline int fused_launches(const tlbm_host::DevState&) {
    return 1;
}

template <int Q, typename S>
inline MGeom mgeom(const tlbm_host::DevState& d, const FusedCfg<Q>& c) {
    MGeom g;
    g.NA = d.nx;
    g.NB = (Q == 19) ? d.ny : 1;
    g.NM = (Q == 19) ? d.nz : d.ny;
    g.rowstride = (long long)d.ncx * Fmt<Q, S>::CHUNK;
    g.NC = (g.NM + c.MC - 1) / c.MC;  // chunks of MC planes or one fewer (balanced)
    g.bytes = d.pop_bytes;
    g.check = d.check;
    g.flag = d.flag;
    g.tilesA = (g.NA + c.TX - 1) / c.TX;
    g.tilesB = (g.NB + c.TY - 1) / c.TY;
    return g;
}

template <int Q, typename S>
inline long long fused_blocks(const tlbm_host::DevState& d) {
    const FusedCfg<Q> c = fused_cfg<Q>(d);
    const MGeom g = mgeom<Q, S>(d, c);
    return (long long)g.tilesA * g.tilesB * g.NC;
}

// Launch with dyn bytes of dynamic shared memory and the smallest shared-memory
// carveout that holds bps blocks per SM, so that the rest of the SM's 256 KB stays
// L1 (which holds the kernel's loads in flight).
template <typename K, typename... Args>
inline cudaError_t launch_smem(K kern, int dyn, int threads, int bps, long long nb, cudaStream_t st, Args... args) {
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (e != cudaSuccess) return e;
    const long long need = (long long)bps * ((long long)fa.sharedSizeBytes + dyn + 1024);
    const int pct = (int)((need * 100 + 233471) / 233472);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct > 100 ? 100 : pct);
    if (e != cudaSuccess) return e;
    kern<<<(int)nb, threads, dyn, st>>>(args...);
    return cudaSuccess;
}
// ... of a D2Q9 kernel with stg staged values per thread of 128
template <typename K, typename... Args>
inline cudaError_t launch_staged(K kern, int stg, long long nb, cudaStream_t st, Args... args) {
    return launch_smem(kern, stg * 2 * 128 * (int)sizeof(float), 128, 4, nb, st, args...);
}
// ... of k_bulk
template <typename S, typename K, typename... Args>
inline cudaError_t launch_bulk(K kern, long long nb, cudaStream_t st, Args... args) {
    using B = BulkShape<S>;
    return launch_smem(kern, B::SMEM, B::THREADS, B::BPS, nb, st, args...);
}

template <int Q, typename S>
inline cudaError_t fused_step(tlbm_host::DevState& d, const Phys<typename Store<S>::T>& P, cudaStream_t st) {
    const FusedCfg<Q> c = fused_cfg<Q>(d);
    const MGeom g = mgeom<Q, S>(d, c);
    const long long nb = (long long)g.tilesA * g.tilesB * g.NC;
    if (nb > 0x7fffffffLL || nb > d.partials_cap) return cudaErrorInvalidConfiguration;
    const S* src = static_cast<const S*>(d.pop[d.cur]);
    S* dst = static_cast<S*>(d.pop[1 - d.cur]);
    if (d.solid && !d.nbm_ready) {
        const Geom gg{d.nx, d.ny, d.nz, d.N, d.Np, d.ncx};
        k_nbmask<Q><<<grid_of(d.N, d.sms), 256, 0, st>>>(gg, d.solid, d.nbm);
        d.nbm_ready = 1;
    }
    if (d.checked) {
        // bounds-checked kernels of the default FP32 tiles (recording, never trapping)
        if constexpr (sizeof(S) == 4) {
            if (!d.check) return cudaErrorInvalidValue;
            if (d.solid) {
                if constexpr (Q == 19) k_fused_solid<Q, S, 32, 4, true><<<(int)nb, 128, 0, st>>>(g, src, dst, d.nbm, P, d.partials);
                else k_fused_solid<Q, S, 128, 1, true><<<(int)nb, 128, 0, st>>>(g, src, dst, d.nbm, P, d.partials);
            } else {
                cudaError_t e;
                if constexpr (Q == 19) e = launch_bulk<S>(k_bulk<S, true>, nb, st, g, src, dst, P, d.partials);
                else e = launch_staged(k_fused_x<Q, S, 128, 1, 27, true>, 27, nb, st, g, src, dst, P, d.partials);
                if (e != cudaSuccess) return e;
            }
            return cudaGetLastError();
        } else {
            return cudaErrorNotSupported;
        }
    }
    if (d.solid) {
        auto gos = [&](auto kern, int threads) {
            kern<<<(int)nb, threads, 0, st>>>(g, src, dst, d.nbm, P, d.partials);
        };
        if constexpr (Q == 19) {
            if constexpr (sizeof(S) == 8) gos(k_fused_solid<Q, S, 16, 4>, 64);
            else gos(k_fused_solid<Q, S, 32, 4>, 128);
        } else {
            if (c.TX == 256) gos(k_fused_solid<Q, S, 256, 1>, 256);
            else if (c.TX == 64) gos(k_fused_solid<Q, S, 64, 1>, 64);
            else if (c.TX == 32) {
                if constexpr (sizeof(S) == 8) gos(k_fused_solid<Q, S, 32, 1>, 32);
            } else gos(k_fused_solid<Q, S, 128, 1>, 128);
        }
        return cudaGetLastError();
    }
    auto go = [&](auto kern, int threads) { kern<<<(int)nb, threads, 0, st>>>(g, src, dst, P, d.partials); };
    if constexpr (sizeof(S) == 8) {
        // double storage is the parity path: one tile shape per lattice and size
        if constexpr (Q == 19) go(k_fused<Q, S, 16, 8, false, false>, 128);
        else if (c.TX == 32) go(k_fused<Q, S, 32, 1, false, false>, 32);
        else go(k_fused<Q, S, 128, 1, false, false>, 128);
    } else if constexpr (Q == 19) {
        const cudaError_t e = launch_bulk<S>(k_bulk<S, false>, nb, st, g, src, dst, P, d.partials);
        if (e != cudaSuccess) return e;
    } else {
        if (c.shape >= 4 && !d.solid) {
            // 128-node rows with staging: 4 the 18 lane-shifted values, 5 (default)
            // all 27, with the per-warp prefetch and evict-first stores and
            // collision loads
            const cudaError_t e =
                c.shape == 4 ? launch_staged(k_fused_x<Q, S, 128, 1, 18>, 18, nb, st, g, src, dst, P, d.partials)
                             : launch_staged(k_fused_x<Q, S, 128, 1, 27>, 27, nb, st, g, src, dst, P, d.partials);
            return e != cudaSuccess ? e : cudaGetLastError();
        }
        if (c.TX == 256) {
            switch (c.mode) {
                case 1: go(k_fused<Q, S, 256, 1, true, false>, 256); break;
                case 2: go(k_fused<Q, S, 256, 1, false, true>, 256); break;
                case 3: go(k_fused<Q, S, 256, 1, true, true>, 256); break;
                default: go(k_fused<Q, S, 256, 1, false, false>, 256);
            }
        } else if (c.TX == 64) {
            go(k_fused<Q, S, 64, 1, false, false>, 64);
        } else if (c.mode == 4) {
            go(k_fused<Q, S, 128, 1, false, false, true>, 128);
        } else if (c.mode == 12) {
            go(k_fused<Q, S, 128, 1, false, false, true, 1>, 128);
        } else if (c.mode == 13) {
            go(k_fused<Q, S, 128, 1, false, false, true, 2>, 128);
        } else {
            go(k_fused<Q, S, 128, 1, false, false>, 128);  // plain loop
        }
    }
    return cudaGetLastError();
}

// ---- batches: every member uses the batch's tile; descriptors for both parities

template <int Q, typename S>
inline cudaError_t batch_build(tlbm_host::BatchState& b, cudaStream_t st) {
    using T = typename Store<S>::T;
    const int n = b.count;
    if (n < 1) return cudaErrorInvalidValue;
    const bool solid = b.sims[0]->solid != nullptr;
    std::vector<SimDesc<T>> h(2 * (size_t)n);
    long long block0 = 0;
    b.auto_tile = b.tile;
    b.narrow = 1;
    for (int k = 0; k < n; ++k) b.narrow = b.narrow && narrow_rows(*b.sims[k]);
    if ((b.tile >> 8) == 0) {
        // members whose own chunks do not fill the device twice keep them; beyond
        // that the halo planes of short chunks are what costs, and one chunk is
        // chosen for the whole grid (24 wells of 128x64 .. 768x384, FP32: 343 us a
        // step with chunks of 4 to 8 planes, see k_fused_solid_batch)
        std::vector<long long> cols, caps;
        long long own = 0;
        std::vector<int> nm;
        FusedCfg<Q> c{};
        tlbm_host::DevState d0 = *b.sims[0];
        for (int k = 0; k < n; ++k) {
            tlbm_host::DevState dd = *b.sims[k];
            dd.tile = b.tile;
            dd.rows128 = !b.narrow;
            own += fused_blocks<Q, S>(dd);
            c = fused_cfg<Q>(dd);
            cols.push_back((long long)((dd.nx + c.TX - 1) / c.TX) * (Q == 19 ? (dd.ny + c.TY - 1) / c.TY : 1));
            nm.push_back(Q == 19 ? dd.nz : dd.ny);
            caps.push_back(dd.partials_cap);
        }
        if (own >= 2LL * c.res(d0) * d0.sms) {
            const int mc = pick_chunk(cols.data(), nm.data(), caps.data(), n, c.halo(d0), c.res(d0), d0.sms, Q == 19,
                                      d0.prec == 0);
            b.auto_tile = (b.tile & 255) | mc << 8;
        }
    }
    for (int k = 0; k < n; ++k) {
        tlbm_host::DevState& d = *b.sims[k];
        if ((d.solid != nullptr) != solid || d.cur != b.sims[0]->cur) return cudaErrorInvalidValue;
        if (solid && !d.nbm_ready) {
            const Geom gg{d.nx, d.ny, d.nz, d.N, d.Np, d.ncx};
            k_nbmask<Q><<<grid_of(d.N, d.sms), 256, 0, st>>>(gg, d.solid, d.nbm);
            d.nbm_ready = 1;
        }
        tlbm_host::DevState dd = d;
        dd.tile = b.auto_tile;
        dd.rows128 = !b.narrow;
        const FusedCfg<Q> c = fused_cfg<Q>(dd);
        // shapes with a batched kernel (batch_step): every solid shape; periodic
        // D3Q19 all but 1 and 2; periodic D2Q9 rows of 128 and the one-warp rows
        const int variant = sizeof(S) == 8 ? 0 : (b.tile & 15);
        const bool shape_ok = solid || (Q == 19 ? variant != 1 && variant != 2 : c.TX == 128 || sizeof(S) == 8);
        if (!shape_ok) return cudaErrorInvalidConfiguration;
        const MGeom g = mgeom<Q, S>(dd, c);
        const long long nb = (long long)g.tilesA * g.tilesB * g.NC;
        if (nb > d.partials_cap) return cudaErrorInvalidConfiguration;
        for (int par = 0; par < 2; ++par) {
            SimDesc<T>& e = h[(size_t)par * n + k];
            e.g = g;
            e.src = d.pop[par];
            e.dst = d.pop[1 - par];
            e.nbm = d.nbm;
            e.P = to_phys<T>(d.phys);
            e.partials = d.partials;
            e.step_mass = d.step_mass;
            e.flag = d.flag;
            e.block0 = (int)block0;
            e.nblocks = (int)nb;
        }
        block0 += nb;
    }
    if (block0 > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    b.blocks = block0;
    cudaError_t e = cudaSuccess;
    if (!b.desc) e = cudaMalloc(&b.desc, sizeof(SimDesc<T>) * 2 * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.desc, h.data(), sizeof(SimDesc<T>) * 2 * (size_t)n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) b.built = 1;
    return e;
}

template <int Q, typename S>
inline cudaError_t batch_step(tlbm_host::BatchState& b, cudaStream_t st, cudaEvent_t ev0 = nullptr,
                              cudaEvent_t ev1 = nullptr) {
    using T = typename Store<S>::T;
    const int n = b.count;
    const int par = b.sims[0]->cur;
    const SimDesc<T>* d = static_cast<const SimDesc<T>*>(b.desc) + (size_t)par * n;
    tlbm_host::DevState probe = *b.sims[0];
    probe.tile = b.auto_tile;
    probe.rows128 = !b.narrow;
    const FusedCfg<Q> c = fused_cfg<Q>(probe);
    const int nb = (int)b.blocks;
    if (ev0) cudaEventRecord(ev0, st);
    if (probe.solid) {
        if constexpr (Q == 19) {
            if constexpr (sizeof(S) == 8) k_fused_solid_batch<Q, S, 16, 4><<<nb, 64, 0, st>>>(d, n);
            else k_fused_solid_batch<Q, S, 32, 4><<<nb, 128, 0, st>>>(d, n);
        } else {
            if (c.TX == 256) k_fused_solid_batch<Q, S, 256, 1><<<nb, 256, 0, st>>>(d, n);
            else if (c.TX == 64) k_fused_solid_batch<Q, S, 64, 1><<<nb, 64, 0, st>>>(d, n);
            else if (c.TX == 32) {
                if constexpr (sizeof(S) == 8) k_fused_solid_batch<Q, S, 32, 1><<<nb, 32, 0, st>>>(d, n);
            } else k_fused_solid_batch<Q, S, 128, 1><<<nb, 128, 0, st>>>(d, n);
        }
    } else {
        if constexpr (Q == 19) {
            if constexpr (sizeof(S) == 8) k_fused_batch<Q, S, 16, 8, false, 0><<<nb, 128, 0, st>>>(d, n);
            else {
                const cudaError_t e = launch_bulk<S>(k_bulk_batch<S>, nb, st, d, n);
                if (e != cudaSuccess) return e;
            }
        } else if (sizeof(S) == 8 && c.TX == 32) {
            if constexpr (sizeof(S) == 8) k_fused_batch<Q, S, 32, 1, false, 0><<<nb, 32, 0, st>>>(d, n);
        } else {
            k_fused_batch<Q, S, 128, 1, true, 2><<<nb, 128, 0, st>>>(d, n);
        }
    }
    if (ev1) cudaEventRecord(ev1, st);
    for (int k = 0; k < n; ++k) b.sims[k]->cur ^= 1;
    return cudaGetLastError();
}

// totals of every member's last batched step (the same sums under both parities)
template <int Q, typename S>
inline cudaError_t batch_totals(tlbm_host::BatchState& b, cudaStream_t st) {
    using T = typename Store<S>::T;
    k_mass_final_batch<T><<<b.count, kThreads, 0, st>>>(static_cast<const SimDesc<T>*>(b.desc));
    return cudaGetLastError();
}

}  // namespace tlbm_dev
