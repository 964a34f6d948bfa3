// tlbm_launch.cuh -- host side of the marching kernels: tiles, chunks, launches and
// batches.
#pragma once

#include <algorithm>
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
// blocks drift apart and only the sum counts.  FP64 is bound by its few FP64 units
// once some five warps share an SM (2.8 us for a warp's collision, 0.75 for its
// moments with the halo), and below that by the latency of a warp's own chain (3.5
// us for either): 64x64 takes one plane a block, walled 256x128 two (seven, the
// choice by operations alone, left 1.7 warps on an SM).
// The constants of FP32 and 16 bits were fitted to kernels with plain loads; against the
// present ones, over 57 lattices (64^2 .. 2048x1024, 40^3 .. 160^2x96, periodic and
// between walls, all storages) and 15 chunks of 1 .. 64 planes, the chosen chunk is the
// fastest to 1 % for 41, within 6 % for 48, and 7 to 15 % off for D3Q19 between walls
// and 256x128 between walls; 40^3, periodic, takes six planes where three are 26 %
// faster (FP32; 16 bits 19 %).  Halving 64 or 16 until 4 blocks per SM are reached, the
// earlier rule, had lost up to 27 % with the kernels it was made for.
// Solid-aware blocks (`solid`) wait for one another's loads less: a plane takes 0.62 +
// 0.095 b' of a full SM's (porous lattices, 5 % solid, FP32 517x391: 2.3, 2.6, 3.1, 3.2 us
// a plane at 1 to 4 blocks; 300x20x20 5.7, 6.3, 8.7 at 1, 2, 4).  By the other curve
// 300x20x20 took seven planes a block, 62.3 us a step; at two it is 52.2.
inline double march_cost(double nb, int mc, int halo, int res, int threads, int sms, bool dbl, bool solid) {
    const double full = (double)res * sms;
    if (dbl) {
        const double per = nb / sms, b = per > 8.0 ? per : (double)(long long)(per + 0.9999);
        const double warps = threads / 32.0;
        const double chain = 3.5 * (2 * mc + halo), units = b * warps * (2.8 * mc + 0.75 * (mc + halo));
        return chain > units ? chain : units;
    }
    const double alone = solid ? 0.62 : 0.25, more = solid ? 0.095 : 0.19;
    auto plane = [&](double b) { return alone + more * 4.0 * b / res; };
    const double rounds = nb / full;
    if (rounds >= 4.0) return (mc + halo) * plane(res) * rounds;
    const double whole = (double)(long long)rounds;
    const double rest = nb - whole * full;
    const double b = (double)(long long)((rest + sms - 1) / sms);
    return (mc + halo) * (whole * plane(res) + (rest > 0 ? plane(b) : 0.0));
}

// cols columns of tiles, each with nm planes to march, of lattice `member`
struct Run {
    long long cols;
    int nm, member;
    bool dirty;
};

// Planes per block of the solid-aware body where clean blocks march mc: a plane of it
// takes about 1.6 times as long and it has four halo planes, and a block that
// outlasts the others is the step's time (sweep of 24 wells: one 60-plane block
// was 260 of 310 us).
inline int dirty_chunk(int mc) { return mc <= 4 ? mc : (mc / 2 - 2 > 4 ? mc / 2 - 2 : 4); }

// Planes per block (chunk) of one marching launch over these runs: the cheapest by
// march_cost whose blocks' sums fit every member (caps).  At most 64 planes in
// 2-D; in 3-D 16 once the grid fills the device eight times over (256^3 FP32: 16
// planes 0.692 of HBM, 24..128 planes 0.66..0.69: blocks that start together share
// their halo rows in L2).
inline int pick_chunk(const std::vector<Run>& runs, const std::vector<long long>& caps, int halo, int res, int threads,
                      int sms, bool three_d, bool dbl, bool solid) {
    double best = 0.0;
    int bmc = 0;
    std::vector<long long> nbs(caps.size());
    for (int mc = three_d ? 2 : 1; mc <= 64; ++mc) {
        double nb = 0.0;
        int used = 0;
        for (long long& v : nbs) v = 0;
        for (const Run& r : runs) {
            const int ch = r.dirty ? dirty_chunk(mc) : mc;
            const int nc = (r.nm + ch - 1) / ch, per = (r.nm + nc - 1) / nc;
            nb += (double)r.cols * nc;
            nbs[(size_t)r.member] += r.cols * nc;
            // the longest block, in planes of the body that most planes need
            const int as = r.dirty && (dbl || !solid) && per == ch ? mc : per;
            used = as > used ? as : used;
        }
        bool fits = true;
        for (size_t k = 0; k < caps.size(); ++k) fits = fits && nbs[k] <= caps[k];
        if (!fits) continue;
        const double c = march_cost(nb, used, halo, res, threads, sms, dbl, solid);
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
    // prologue planes a block recomputes, and blocks per SM of the kernel that has the
    // lattice to itself (mixed: of work items)
    int halo(const tlbm_host::DevState& d) const { return d.solid || d.coupling ? 4 : 2; }
    int res(const tlbm_host::DevState& d, bool mixed = false) const {
        if (Q == 19 && d.prec != 0 && !d.solid && !d.coupling) return d.prec == 1 ? BulkShape<float>::BPS : BulkShape<__half>::BPS;  // k_bulk
        if (Q == 19 && d.prec != 0 && d.solid && !mixed) return 3;  // k_fused_solid
        return d.prec == 0 && TX == 32 ? 8 : 512 / (TX * TY);
    }
};

// d.tile = shape | mode << 4 | chunk << 8: shape 0 = default.  D3Q19 has one tile per
// storage format (FP32 and 16-bit: k_bulk, 32x4 nodes; double: k_fused, 16x8), and
// D2Q9 in FP32 and 16 bits one kernel on rows of 128 nodes (k_bulk2; shape 2: 256,
// 3: 64).  The other shapes and the modes are accepted and change nothing.  chunk =
// planes per block (0 = pick_chunk).
// D2Q9 in double: rows of 32 nodes (one warp) where rows of 128 in chunks of four
// planes leave SMs idle; wider rows recompute fewer halo moments.
// Where the blocks' sums do not fit the scratch on narrow rows (a short given chunk; a
// single row of more than 38912 nodes at any chunk) rows of 128 are taken.  A batch
// launches one tile for all members: narrow only if every member is.
inline bool narrow_rows(const tlbm_host::DevState& d) {
    if (d.rows != 0) return d.rows == 32;
    const int mc = (d.tile >> 8) ? d.tile >> 8 : 64;  // pick_chunk's longest
    return d.N < 512LL * d.sms && (long long)((d.nx + 31) / 32) * ((d.ny + mc - 1) / mc) <= d.partials_cap;
}

template <int Q>
inline FusedCfg<Q> fused_cfg(const tlbm_host::DevState& d) {
    const bool dbl = d.prec == 0;  // double storage: one default shape only
    const int tile = d.checked ? 0 : d.tile;  // the checked kernels use the default tile
    const int variant = dbl ? 0 : (tile & 15);
    int mc = tile >> 8;
    FusedCfg<Q> c{};
    if (d.coupling) {
        c.TX = Q == 19 ? (dbl ? 16 : 32) : 128;  // k_guo_fused
        c.TY = Q == 19 ? (dbl ? 4 : 8) : 1;
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
        c.TX = dbl ? (narrow_rows(d) ? 32 : 128) : (variant == 2 ? 256 : (variant == 3 ? 64 : 128));  // k_bulk2
        c.TY = 1;
    }
    const int NA = d.nx;
    const int NB = (Q == 19) ? d.ny : 1;
    const int NM = (Q == 19) ? d.nz : d.ny;
    if (Q == 19 && mc > 0 && !dbl && !d.solid && !d.coupling && (variant == 1 || variant == 2)) {
        // shapes 1 and 2 name tiles of 32x8 and 64x4 nodes: a chunk whose sums fit the
        // scratch on those is doubled until they fit on 32x4
        auto nb = [&](int tx, int ty, int ch) {
            return (long long)((NA + tx - 1) / tx) * ((NB + ty - 1) / ty) * ((NM + ch - 1) / ch);
        };
        if (nb(variant == 2 ? 64 : 32, variant == 1 ? 8 : 4, mc) <= d.partials_cap)
            while (mc < NM && nb(32, 4, mc) > d.partials_cap) mc *= 2;
    }
    if (mc <= 0) {
        const long long cols = (long long)((NA + c.TX - 1) / c.TX) * ((NB + c.TY - 1) / c.TY);
        mc = pick_chunk({Run{cols, NM, 0, false}}, {d.partials_cap}, c.halo(d), c.res(d), c.TX * c.TY, d.sms, Q == 19, dbl,
                        d.solid != nullptr);
    }
    c.MC = mc < 1 ? 1 : (mc > NM ? NM : mc);
    return c;
}

// ---- lattices with solid nodes: the blocks' work

// A column's planes as runs of one kind: dirty planes have a solid node within two
// nodes of the tile (ghosts of the one-node halo need moments of the second, whose
// pulls a solid node turns back); planes whose tile nodes are all solid are left
// out.  Clean gaps shorter than four planes join their dirty neighbours (each
// block has 2 (clean) or 4 (dirty) halo planes to recompute).
struct ColumnRun {
    int A0, B0, m0, nm;
    bool dirty;
};

// d.units[(m NB + b) ncx + u], for 32 nodes u of row b, plane m: bit 0 a solid node
// in x from two before to two behind, bit 1 all of them solid.
template <int Q>
inline std::vector<ColumnRun> column_runs(const tlbm_host::DevState& d, const FusedCfg<Q>& c) {
    const int NB = Q == 19 ? d.ny : 1, NM = Q == 19 ? d.nz : d.ny, HB = Q == 19 ? 2 : 0;
    std::vector<ColumnRun> out;
    auto around = [](int v, int n) {  // periodic; without a division for every node
        while (v < 0) v += n;
        while (v >= n) v -= n;
        return v;
    };
    std::vector<unsigned char> near((size_t)NM), full((size_t)NM), kind((size_t)NM);
    for (int B0 = 0; B0 < NB; B0 += c.TY)
        for (int A0 = 0; A0 < d.nx; A0 += c.TX) {
            const int u0 = A0 / 32, u1 = (A0 + c.TX + 31) / 32 < d.ncx ? (A0 + c.TX + 31) / 32 : d.ncx;
            for (int m = 0; m < NM; ++m) {
                unsigned char any = 0, all = 1;
                for (int b = B0 - HB; b < B0 + c.TY + HB; ++b) {
                    const bool tile = b >= B0 && b < B0 + c.TY && b < NB;
                    const unsigned char* row = d.units + ((size_t)m * NB + (size_t)around(b, NB)) * d.ncx;
                    for (int u = u0; u < u1; ++u) {
                        any |= row[u] & 1;
                        if (tile && !(row[u] & 2)) all = 0;
                    }
                }
                near[(size_t)m] = any;
                full[(size_t)m] = all;
            }
            for (int m = 0; m < NM; ++m) {
                unsigned char any = 0;
                for (int k = -2; k <= 2; ++k) any |= near[(size_t)around(m + k, NM)];
                kind[(size_t)m] = full[(size_t)m] ? 2 : any;
            }
            for (int m = 0; m < NM;) {  // short clean gaps
                int e = m;
                while (e < NM && kind[(size_t)e] == 0) ++e;
                if (e > m && e - m < 4 && e - m < NM)
                    for (int k = m; k < e; ++k) kind[(size_t)k] = 1;
                m = e > m ? e : m + 1;
            }
            for (int m = 0; m < NM;) {
                int e = m + 1;
                while (e < NM && kind[(size_t)e] == kind[(size_t)m]) ++e;
                if (kind[(size_t)m] != 2) out.push_back(ColumnRun{A0, B0, m, e - m, kind[(size_t)m] == 1});
                m = e;
            }
        }
    return out;
}

// Whether an engine's solid lattice is stepped by work items: D2Q9 always (k_mix);
// D3Q19 (FP32, 16-bit: dirty blocks by k_fused_solid, clean ones by k_bulk, two
// launches side by side) where the clean blocks alone fill the device.
template <int Q>
inline bool wants_items(const tlbm_host::DevState& d) {
    return d.solid && d.units && (Q == 9 || d.prec != 0);
}

// The work items (A0, B0, M0, 2 M1 + dirty) of chunk mc, dirty ones first: they take
// longest.  Returns the number of dirty ones.
inline int make_items(const std::vector<ColumnRun>& runs, int mc, std::vector<int4>& out) {
    int dirty = 0;
    for (int pass = 1; pass >= 0; --pass) {
        const size_t first = out.size();
        for (const ColumnRun& r : runs) {
            if (r.dirty != (pass == 1)) continue;
            const int ch = r.dirty ? dirty_chunk(mc) : mc, nc = (r.nm + ch - 1) / ch;
            for (int c = 0; c < nc; ++c)
                out.push_back(make_int4(r.A0, r.B0, r.m0 + (int)((long long)c * r.nm / nc),
                                        2 * (r.m0 + (int)((long long)(c + 1) * r.nm / nc)) + pass));
        }
        // blocks that start together work on neighbouring planes and share rows in L2
        std::stable_sort(out.begin() + (long)first, out.end(), [](const int4& a, const int4& b) { return a.z < b.z; });
        if (pass == 1) dirty = (int)out.size();
    }
    return dirty;
}

inline int runs_halo(const std::vector<ColumnRun>& runs) {
    long long d = 0, c = 0;
    for (const ColumnRun& r : runs) (r.dirty ? d : c) += r.nm;
    return c > d ? 2 : 4;
}

inline void add_runs(const std::vector<ColumnRun>& runs, int member, std::vector<Run>& out) {
    for (const ColumnRun& r : runs) out.push_back(Run{1, r.nm, member, r.dirty});
}

// Work items of an engine's lattice at its tile and chunk; none where one grid over
// the whole lattice serves (ndirty = 0, out empty).
template <int Q, typename S>
inline int solid_items(const tlbm_host::DevState& d, std::vector<int4>& out) {
    out.clear();
    if (!wants_items<Q>(d)) return 0;
    tlbm_host::DevState dd = d;
    dd.rows = narrow_rows(d) ? 32 : 128;
    dd.tile = d.tile | ((d.tile >> 8) ? 0 : 1 << 8);  // any chunk: only the tile is wanted
    const FusedCfg<Q> c = fused_cfg<Q>(dd);
    const std::vector<ColumnRun> runs = column_runs<Q>(d, c);
    int mc = d.tile >> 8;
    if (mc == 0) {
        std::vector<Run> all;
        add_runs(runs, 0, all);
        const int halo = runs_halo(runs);
        mc = pick_chunk(all, {d.partials_cap}, halo, c.res(d, true), c.TX * c.TY, d.sms, Q == 19, d.prec == 0, halo == 4);
    }
    int dirty = make_items(runs, mc, out);
    const long long clean = (long long)out.size() - dirty;
    if ((long long)out.size() > d.partials_cap || (Q == 19 && clean < 2LL * d.sms)) {
        out.clear();
        dirty = 0;
    }
    return dirty;
}

// Whether a step takes the engine's work items.  A checked step runs on the default
// tile: it takes them where they are of its row width (a chunk of its own is no matter,
// the items hold their planes), and else one grid.
template <int Q>
inline bool use_items(const tlbm_host::DevState& d) {
    return d.nitems > 0 && (!d.checked || Q == 19 || ((d.tile & 15) != 2 && (d.tile & 15) != 3));
}

template <int Q, typename S>
inline bool fused_supported(const tlbm_host::DevState& d) {
    return d.solid == nullptr || d.nbm != nullptr;
}

template <int Q, typename S>
inline int fused_launches(const tlbm_host::DevState& d) {
    return Q == 19 && use_items<Q>(d) && d.ndirty > 0 ? 2 : 1;
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
    g.items = use_items<Q>(d) ? static_cast<const int4*>(d.items) : nullptr;
    g.tilesA = (g.NA + c.TX - 1) / c.TX;
    g.tilesB = (g.NB + c.TY - 1) / c.TY;
    return g;
}

template <int Q, typename S>
inline long long fused_blocks(const tlbm_host::DevState& d) {
    if (use_items<Q>(d)) return d.nitems;
    const FusedCfg<Q> c = fused_cfg<Q>(d);
    const MGeom g = mgeom<Q, S>(d, c);
    return (long long)g.tilesA * g.tilesB * g.NC;
}

// Where a kernel goes: its stream, and whether it may start while the one before it on
// that stream still runs.
struct At {
    cudaStream_t st;
    bool early = true;
    At(cudaStream_t s, bool e = true) : st(s), early(e) {}
};

// Launch of a step kernel (grid_ready) with dyn bytes of dynamic shared memory.
template <typename K, typename... Args>
inline cudaError_t launch_step(K kern, int dyn, int threads, long long nb, At at, Args... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)nb);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = (size_t)dyn;
    c.stream = at.st;
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = at.early ? 1 : 0;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, args...);
}
// The same with the smallest shared-memory
// carveout that holds bps blocks per SM, so that the rest of the SM's 256 KB stays
// L1 (which holds the kernel's loads in flight).
template <typename K, typename... Args>
inline cudaError_t launch_smem(K kern, int dyn, int threads, int bps, long long nb, At at, Args... args) {
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (e != cudaSuccess) return e;
    const long long need = (long long)bps * ((long long)fa.sharedSizeBytes + dyn + 1024);
    const int pct = (int)((need * 100 + 233471) / 233472);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct > 100 ? 100 : pct);
    if (e != cudaSuccess) return e;
    return launch_step(kern, dyn, threads, nb, at, args...);
}
// ... of k_bulk2
template <typename S, int TX, typename K, typename... Args>
inline cudaError_t launch_bulk2(K kern, long long nb, At at, Args... args) {
    return launch_smem(kern, Bulk2Shape<S, TX>::SMEM, TX, 512 / TX, nb, at, args...);
}
// ... of k_bulk
template <typename S, typename K, typename... Args>
inline cudaError_t launch_bulk(K kern, long long nb, At at, Args... args) {
    using B = BulkShape<S>;
    return launch_smem(kern, B::SMEM, B::THREADS, B::BPS, nb, at, args...);
}

// One step of a lattice with solid nodes: work items, or one grid of solid-aware blocks.
// CHK: the bounds-checked kernels, at the default tile.
template <int Q, typename S, bool CHK>
inline cudaError_t solid_step(tlbm_host::DevState& d, const FusedCfg<Q>& c, const MGeom& g, long long nb, const S* src,
                              S* dst, const Phys<typename Store<S>::T>& P, cudaStream_t st) {
    if (nb == 0) return cudaSuccess;  // no fluid node
    cudaError_t e = cudaSuccess;
    if constexpr (Q == 19) {
        constexpr int TX = sizeof(S) == 8 ? 16 : 32;
        const long long nd = use_items<Q>(d) ? d.ndirty : nb;
        // dirty and clean blocks side by side: the clean ones' launch on a second
        // stream, between an event behind the step before and one that the next
        // step waits for.  (Both on one stream, the second launch not waiting for
        // the first, read the step before without a dependency of their own, and
        // were no faster: 144x128x80 FP32 210 us a step, 206 with the events.)
        const bool fork = nd > 0 && nb > nd;
        if (fork) {
            e = cudaEventRecord(d.forked, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(d.side, d.forked, 0);
        }
        auto dirty = [&](auto kern, int bps) {
            return launch_smem(kern, solid_smem<Q, S>(TX, 4), TX * 4, bps, nd, At(st, !fork), g, src, dst, d.nbm, P, d.partials);
        };
        if (e == cudaSuccess && nd > 0) {
            if constexpr (sizeof(S) < 8 && !CHK)
                e = fork ? dirty(k_fused_solid<Q, S, TX, 4>, 4) : dirty(k_fused_solid<Q, S, TX, 4, false, 3>, 3);
            else e = dirty(k_fused_solid<Q, S, TX, 4, CHK>, 512 / (TX * 4));
        }
        if constexpr (sizeof(S) < 8) {
            if (e == cudaSuccess && nb > nd) {
                MGeom gc = g;
                gc.items = g.items + nd;
                e = launch_bulk<S>(k_bulk<S, CHK>, nb - nd, At(fork ? d.side : st, !fork), gc, src, dst, P,
                                   d.partials + 3 * nd);
            }
        }
        if (fork) {
            const cudaError_t e1 = cudaEventRecord(d.joined, d.side), e2 = cudaStreamWaitEvent(st, d.joined, 0);
            if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2;
        }
    } else {
        auto mix = [&](auto kern, int TX, int dyn) {
            e = launch_smem(kern, dyn, TX, blocks_per_sm<S>(TX), nb, st, g, src, dst, d.nbm, P, d.partials);
        };
        if constexpr (CHK) {
            mix(k_mix<Q, S, 128, true>, 128, Mix<Q, S>::template smem<128>());
        } else if constexpr (sizeof(S) == 8) {
            if (c.TX == 32) mix(k_mix<Q, S, 32>, 32, Mix<Q, S>::template smem<32>());
            else mix(k_mix<Q, S, 128>, 128, Mix<Q, S>::template smem<128>());
        } else {
            if (c.TX == 256) mix(k_mix<Q, S, 256>, 256, Mix<Q, S>::template smem<256>());
            else if (c.TX == 64) mix(k_mix<Q, S, 64>, 64, Mix<Q, S>::template smem<64>());
            else mix(k_mix<Q, S, 128>, 128, Mix<Q, S>::template smem<128>());
        }
    }
    return e;
}

template <int Q, typename S>
inline cudaError_t fused_step(tlbm_host::DevState& d, const Phys<typename Store<S>::T>& P, cudaStream_t st) {
    const FusedCfg<Q> c = fused_cfg<Q>(d);
    const MGeom g = mgeom<Q, S>(d, c);
    const long long nb = fused_blocks<Q, S>(d);
    if (nb > 0x7fffffffLL || nb > d.partials_cap) return cudaErrorInvalidConfiguration;
    const S* src = static_cast<const S*>(d.pop[d.cur]);
    S* dst = static_cast<S*>(d.pop[1 - d.cur]);
    if (d.solid && !d.nbm_ready) {
        const Geom gg{d.nx, d.ny, d.nz, d.N, d.Np, d.ncx};
        k_nbmask<Q><<<grid_of(d.N, d.sms), 256, 0, st>>>(gg, d.solid, d.nbm);
        d.nbm_ready = 1;
    }
    cudaError_t e = cudaSuccess;
    if (d.checked) {
        // bounds-checked kernels of the default FP32 tiles (recording, never trapping)
        if constexpr (sizeof(S) == 4) {
            if (!d.check) return cudaErrorInvalidValue;
            if (d.solid) e = solid_step<Q, S, true>(d, c, g, nb, src, dst, P, st);
            else if constexpr (Q == 19) e = launch_bulk<S>(k_bulk<S, true>, nb, st, g, src, dst, P, d.partials);
            else e = launch_bulk2<S, 128>(k_bulk2<S, 128, true>, nb, st, g, src, dst, P, d.partials);
            return e != cudaSuccess ? e : cudaGetLastError();
        } else {
            return cudaErrorNotSupported;
        }
    }
    if (d.solid) {
        e = solid_step<Q, S, false>(d, c, g, nb, src, dst, P, st);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    if constexpr (sizeof(S) == 8) {
        // double storage is the parity path: one tile shape per lattice and size
        auto go = [&](auto kern, int threads) {
            e = launch_step(kern, fused_smem<Q, S>(c.TX, c.TY), threads, nb, st, g, src, dst, P, d.partials);
        };
        if constexpr (Q == 19) go(k_fused<Q, S, 16, 8>, 128);
        else if (c.TX == 32) go(k_fused<Q, S, 32, 1>, 32);
        else go(k_fused<Q, S, 128, 1>, 128);
    } else if constexpr (Q == 19) {
        e = launch_bulk<S>(k_bulk<S, false>, nb, st, g, src, dst, P, d.partials);
    } else {
        if (c.TX == 256) e = launch_bulk2<S, 256>(k_bulk2<S, 256, false>, nb, st, g, src, dst, P, d.partials);
        else if (c.TX == 64) e = launch_bulk2<S, 64>(k_bulk2<S, 64, false>, nb, st, g, src, dst, P, d.partials);
        else e = launch_bulk2<S, 128>(k_bulk2<S, 128, false>, nb, st, g, src, dst, P, d.partials);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
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
    for (int k = 0; k < n; ++k) {
        tlbm_host::DevState dd = *b.sims[k];
        dd.tile = b.tile;
        b.narrow = b.narrow && narrow_rows(dd);
    }
    // tile of member k (chunk 1 stands for any), its runs and its blocks with chunk 0
    // (its own choice) or mc
    auto member = [&](int k, int mc) {
        tlbm_host::DevState dd = *b.sims[k];
        dd.tile = (b.tile & 255) | mc << 8;
        dd.rows = b.narrow ? 32 : 128;
        dd.items = nullptr;
        dd.nitems = 0;
        return dd;
    };
    std::vector<std::vector<int4>> items((size_t)n);
    auto blocks = [&](int k, const tlbm_host::DevState& dd) -> long long {
        if (Q == 9 && solid) {
            solid_items<Q, S>(dd, items[(size_t)k]);
            if (!items[(size_t)k].empty()) return (long long)items[(size_t)k].size();
        }
        return fused_blocks<Q, S>(dd);
    };
    if ((b.tile >> 8) == 0) {
        // members whose own chunks fit the device at once keep them; beyond that a few
        // blocks of a second round, and then the halo planes of short chunks, are what
        // costs, and one chunk is chosen for the whole grid (24 wells of 128x64 ..
        // 768x384, FP32: 343 us a step with chunks of 4 to 8 planes)
        std::vector<Run> runs;
        std::vector<long long> caps;
        long long own = 0;
        const tlbm_host::DevState d0 = member(0, 1);
        FusedCfg<Q> c{};
        int halo = 0;
        for (int k = 0; k < n; ++k) {
            own += blocks(k, member(k, 0));
            const tlbm_host::DevState dd = member(k, 1);
            c = fused_cfg<Q>(dd);
            if (Q == 9 && solid) {
                const std::vector<ColumnRun> cr = column_runs<Q>(dd, c);
                add_runs(cr, k, runs);
                halo += runs_halo(cr);
            } else {
                runs.push_back(Run{(long long)((dd.nx + c.TX - 1) / c.TX) * (Q == 19 ? (dd.ny + c.TY - 1) / c.TY : 1),
                                   Q == 19 ? dd.nz : dd.ny, k, false});
                halo += c.halo(dd);
            }
            caps.push_back(dd.partials_cap);
        }
        if (own > (long long)c.res(d0, true) * d0.sms) {
            halo = (halo + n / 2) / n;
            const int mc = pick_chunk(runs, caps, halo, c.res(d0, true), c.TX * c.TY, d0.sms, Q == 19, d0.prec == 0,
                                      solid && halo == 4);
            b.auto_tile = (b.tile & 255) | mc << 8;
        }
    }
    size_t nit = 0;
    std::vector<long long> nbs((size_t)n);
    for (int k = 0; k < n; ++k) {
        nbs[(size_t)k] = blocks(k, member(k, b.auto_tile >> 8));
        nit += items[(size_t)k].size();
    }
    cudaError_t e = cudaSuccess;
    if (nit > 0) {
        e = cudaStreamSynchronize(st);  // no step in flight reads the items that are replaced
        if (e == cudaSuccess && b.items) e = cudaFree(b.items);
        b.items = nullptr;
        if (e == cudaSuccess) e = cudaMalloc(&b.items, sizeof(int4) * nit);
        if (e != cudaSuccess) return e;
    }
    size_t it0 = 0;
    for (int k = 0; k < n; ++k) {
        tlbm_host::DevState& d = *b.sims[k];
        if ((d.solid != nullptr) != solid || d.cur != b.sims[0]->cur) return cudaErrorInvalidValue;
        if (solid && !d.nbm_ready) {
            const Geom gg{d.nx, d.ny, d.nz, d.N, d.Np, d.ncx};
            k_nbmask<Q><<<grid_of(d.N, d.sms), 256, 0, st>>>(gg, d.solid, d.nbm);
            d.nbm_ready = 1;
        }
        const tlbm_host::DevState dd = member(k, b.auto_tile >> 8);
        const FusedCfg<Q> c = fused_cfg<Q>(dd);
        // shapes with a batched kernel (batch_step): every solid shape; periodic
        // D3Q19 all but 1 and 2; periodic D2Q9 rows of 128 and the one-warp rows
        const int variant = sizeof(S) == 8 ? 0 : (b.tile & 15);
        const bool shape_ok = solid || (Q == 19 ? variant != 1 && variant != 2 : c.TX == 128 || sizeof(S) == 8);
        if (!shape_ok) return cudaErrorInvalidConfiguration;
        MGeom g = mgeom<Q, S>(dd, c);
        const long long nb = nbs[(size_t)k];
        if (nb > d.partials_cap || nb < 1) return cudaErrorInvalidConfiguration;
        if (!items[(size_t)k].empty()) {
            int4* to = static_cast<int4*>(b.items) + it0;
            e = cudaMemcpyAsync(to, items[(size_t)k].data(), sizeof(int4) * items[(size_t)k].size(), cudaMemcpyHostToDevice, st);
            if (e != cudaSuccess) return e;
            g.items = to;
            it0 += items[(size_t)k].size();
        }
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
    if (!b.desc) e = cudaMalloc(&b.desc, sizeof(SimDesc<T>) * 2 * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.desc, h.data(), sizeof(SimDesc<T>) * 2 * (size_t)n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
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
    probe.rows = b.narrow ? 32 : 128;
    const FusedCfg<Q> c = fused_cfg<Q>(probe);
    const int nb = (int)b.blocks;
    if (ev0) cudaEventRecord(ev0, st);
    cudaError_t e = cudaSuccess;
    if (probe.solid) {
        if constexpr (Q == 19) {
            constexpr int TX = sizeof(S) == 8 ? 16 : 32;
            e = launch_smem(k_fused_solid_batch<Q, S, TX, 4>, solid_smem<Q, S>(TX, 4), TX * 4, 512 / (TX * 4), nb, st, d, n);
        } else {
            auto mix = [&](auto kern, int TX, int dyn) {
                e = launch_smem(kern, dyn, TX, blocks_per_sm<S>(TX), nb, st, d, n);
            };
            if constexpr (sizeof(S) == 8) {
                if (c.TX == 32) mix(k_fused_solid_batch<Q, S, 32, 1>, 32, Mix<Q, S>::template smem<32>());
                else mix(k_fused_solid_batch<Q, S, 128, 1>, 128, Mix<Q, S>::template smem<128>());
            } else {
                if (c.TX == 256) mix(k_fused_solid_batch<Q, S, 256, 1>, 256, Mix<Q, S>::template smem<256>());
                else if (c.TX == 64) mix(k_fused_solid_batch<Q, S, 64, 1>, 64, Mix<Q, S>::template smem<64>());
                else mix(k_fused_solid_batch<Q, S, 128, 1>, 128, Mix<Q, S>::template smem<128>());
            }
        }
    } else {
        auto go = [&](auto kern, int threads) {
            e = launch_smem(kern, fused_smem<Q, S>(c.TX, c.TY), threads, blocks_per_sm<S>(threads), nb, st, d, n);
        };
        if constexpr (Q == 19) {
            if constexpr (sizeof(S) == 8) go(k_fused_batch<Q, S, 16, 8>, 128);
            else e = launch_bulk<S>(k_bulk_batch<S>, nb, st, d, n);
        } else if constexpr (sizeof(S) == 8) {
            if (c.TX == 32) go(k_fused_batch<Q, S, 32, 1>, 32);
            else go(k_fused_batch<Q, S, 128, 1>, 128);
        } else {
            e = launch_bulk2<S, 128>(k_fused_batch<Q, S, 128, 1>, nb, st, d, n);
        }
    }
    if (e != cudaSuccess) return e;
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
