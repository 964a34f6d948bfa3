// tlbm_fused.cuh -- one-kernel time step of the ternary free-energy LB method
// (Semprebon, Krueger, Kusumaatmaja, arXiv:1511.02155): the periodic step in double
// (the other storages bring the same march's populations by bulk copies,
// tlbm_bulk.cuh) and the solid-aware step in every storage.
//
// The equilibria at r need gradients and Laplacians of rho, phi, psi at the
// same time level, i.e. the moments of r's neighbours, which depend on the
// neighbours' populations.  Instead of writing moment arrays to HBM and
// reading the populations twice, each block owns a column of the lattice
// (a TX x TY tile of the in-plane axes) and marches along the last axis
// (z for D3Q19, y for D2Q9) over a chunk of MC planes:
//
//   prologue: moments of planes m0-1 and m0 (tile + one-node halo) -> smem
//   for each plane m of the chunk:
//     M: pull populations of plane m+1 over tile + halo, reduce them to
//        rho, phi, psi (and j = rho u on the tile) into a shared ring
//     __syncthreads
//     C: for each tile node of plane m: gradients and Laplacians from the
//        ring (planes m-1, m, m+1), local thermodynamics, equilibria,
//        BGK, and the store of x*(r) -- populations are pulled again
//        (L1/L2 hits: phase M read them one iteration earlier).
//
// The moment ring has four slots and the j ring three, so one barrier per
// plane suffices (a fast warp writing plane m+2 never touches a slot that a
// slow warp still reads for plane m).  HBM traffic per node is one read and one
// write of the 3Q populations plus the halo's share (about 2/MC extra planes).
#pragma once

#include "tlbm_kernels.cuh"
#include "tlbm_node.cuh"

namespace tlbm_dev {

// velocity components in (in-plane a, in-plane b, marching m) coordinates
template <int Q>
struct Axes {
    static constexpr int D = Lat<Q>::D;
    __host__ __device__ static constexpr int ca(int i) { return Lat<Q>::cx(i); }
    __host__ __device__ static constexpr int cb(int i) { return D == 3 ? Lat<Q>::cy(i) : 0; }
    __host__ __device__ static constexpr int cm(int i) { return D == 3 ? Lat<Q>::cz(i) : Lat<Q>::cy(i); }
};

struct MGeom {
    int NA, NB, NM;       // extents along a, b, m
    int NC;               // chunks along m; chunk c holds planes [c NM / NC, (c+1) NM / NC)
    int tilesA, tilesB;   // tiles per plane
    long long rowstride;  // bytes between consecutive (b, m) rows: ncx * chunk bytes
    long long bytes;      // bytes of one population buffer (bounds-checked kernels)
    unsigned long long* check;  // first bounds violation (bounds-checked kernels)
    int* flag;            // raised by a block whose sums are not finite
    const int4* items;    // lattices with solid nodes: the blocks' work (Work), else null
};

// Steps are launched with programmatic stream serialisation: a step's blocks may be
// placed, and compute their indices, while the step before still runs.  Every
// kernel waits here before its first access to anything that a step writes, and
// then lets the next step's launch begin (not before, so that only one step is ever
// ahead).  The gap between two steps was 2 to 3 us of 13 on a 512x256 lattice.
__device__ __forceinline__ void grid_ready() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One block's share of a march: the tile at (A0, B0), planes M0 .. M1 - 1.
struct Work {
    int A0, B0, M0, M1;
    bool dirty;  // solid nodes within two nodes of the tile: the solid-aware body
};
template <int TX, int TY>
__device__ __forceinline__ Work work_of(const MGeom& g, int bid) {
    if (g.items) {
        const int4 it = g.items[bid];
        return Work{it.x, it.y, it.z, it.w >> 1, (it.w & 1) != 0};
    }
    const int rest = bid / g.tilesA, chunk = rest / g.tilesB;
    return Work{(bid % g.tilesA) * TX, (rest % g.tilesB) * TY, (int)((long long)chunk * g.NM / g.NC),
                (int)((long long)(chunk + 1) * g.NM / g.NC), true};
}

// a block's FP64 sums of rho, phi, psi: its partial sums and the non-finite flag
__device__ __forceinline__ void put_block_sums(const MGeom& g, double* __restrict__ partials, int bid, double r,
                                               double p, double s) {
    partials[3 * bid + 0] = r;
    partials[3 * bid + 1] = p;
    partials[3 * bid + 2] = s;
    if (!(isfinite(r) && isfinite(p) && isfinite(s))) atomicOr(g.flag, 1);
}

// Bounds checks of the checked kernel variants (CHK).  A violation is recorded
// as (code << 56 | offset) in *g.check -- the first one wins -- and the access
// is redirected to a valid address; nothing traps.  Codes: 1 pull source,
// 2 bounce-back source, 3 store target, 4 moment-ring index or offset in a slot of
// bulk copies, 5 mask index.
__device__ __forceinline__ void chk_record(const MGeom& g, unsigned code, long long v) {
    atomicCAS(g.check, 0ull, ((unsigned long long)code << 56) | ((unsigned long long)v & 0x00ffffffffffffffull));
}
// a node pointer (chunk + lane * ESZ) of a population buffer starting at base
template <int Q, typename S, bool CHK, typename P>
__device__ __forceinline__ P* chk_node(const MGeom& g, P* base, P* p, unsigned code) {
    if constexpr (CHK) {
        const long long off = (const unsigned char*)p - (const unsigned char*)base;
        if (off < 0 || off >= g.bytes || (off % Fmt<Q, S>::CHUNK) >= 32LL * Fmt<Q, S>::ESZ) {
            chk_record(g, code, off);
            return base;
        }
    }
    return p;
}
// bytes of a population buffer starting at base that one copy reads
template <bool CHK>
__device__ __forceinline__ const unsigned char* chk_span(const MGeom& g, const unsigned char* base, const unsigned char* p,
                                                         unsigned bytes, unsigned code) {
    if constexpr (CHK) {
        const long long off = p - base;
        if (off < 0 || off + bytes > g.bytes) {
            chk_record(g, code, off);
            return base;
        }
    }
    return p;
}
// an index into an array of n entries
template <bool CHK>
__device__ __forceinline__ long long chk_index(const MGeom& g, long long i, long long n, unsigned code) {
    if constexpr (CHK) {
        if (i < 0 || i >= n) {
            chk_record(g, code, i);
            return 0;
        }
    }
    return i;
}

// blocks per SM asked of the compiler: 16 warps; one-warp blocks in double keep up
// to 255 registers
template <typename S>
constexpr int blocks_per_sm(int threads) {
    return sizeof(S) == 8 && threads == 32 ? 8 : 512 / threads;
}

__device__ __forceinline__ int modp(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// single periodic wrap of v in [-n, 2n)
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }


// Mass totals (rho, phi, psi of the step's input state) of the nodes a thread
// collides, given rd (rho, or rho - 1 where f is stored as f_i - w_i), phi, psi.
// PAIR false sums in double, as the other kernels do.  PAIR true (16-bit formats, and
// FP32 on D2Q9) keeps per quantity a pair (hi, lo) updated by Knuth's TwoSum, and rho as
// the node count plus the summed deviations: no FP64 instruction runs per node, and
// the pairs become doubles once per block; 1-2 % faster.  Its low words round in 24 bits
// themselves, so sums of values far apart hold fewer bits than a double: FP32 on D3Q19
// keeps the double sums.
template <typename T, bool PAIR>
struct MassSum {
    double r = 0.0, p = 0.0, s = 0.0;
    __device__ __forceinline__ void add(double rho, T phi, T psi) {  // rho: rho_total of rd
        r += rho;
        p += (double)phi;
        s += (double)psi;
    }
    __device__ __forceinline__ void get(double& a, double& b, double& c) const {
        a = r;
        b = p;
        c = s;
    }
};
template <>
struct MassSum<float, true> {
    float h[3] = {0.0f, 0.0f, 0.0f}, l[3] = {0.0f, 0.0f, 0.0f};
    int n = 0;
    __device__ __forceinline__ void acc(int c, float x) {
        const float sum = h[c] + x;
        const float bp = sum - h[c];
        l[c] += (h[c] - (sum - bp)) + (x - bp);  // the rounding error of h + x, exactly
        h[c] = sum;
    }
    __device__ __forceinline__ void add(float rd, float phi, float psi) {  // rd = rho - 1 (offset formats)
        acc(0, rd);
        acc(1, phi);
        acc(2, psi);
        ++n;
    }
    __device__ __forceinline__ void get(double& a, double& b, double& c) const {
        a = (double)n + ((double)h[0] + (double)l[0]);
        b = (double)h[1] + (double)l[1];
        c = (double)h[2] + (double)l[2];
    }
};

// bytes of fused_body's moment ring (four planes, tile and one-node halo) and of
// its dynamic shared memory
template <int Q, typename S>
__host__ __device__ constexpr int ring_bytes(int TX, int TY) {
    const int n = 4 * 3 * (TX + 2) * (TY + (Q == 19 ? 2 : 0)) * (int)sizeof(typename Store<S>::T);
    return (n + 15) / 16 * 16;
}
template <int Q, typename S>
__host__ __device__ constexpr int fused_smem(int TX, int TY) {
    return ring_bytes<Q, S>(TX, TY);
}

template <int Q, typename S, int TX, int TY>
__device__ __forceinline__ void fused_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                           const Phys<typename Store<S>::T>& P, double* __restrict__ partials,
                                           const int bid, const Work w) {
    using T = typename Store<S>::T;
    using A = Axes<Q>;
    extern __shared__ __align__(16) unsigned char tlbm_smem[];
    static_assert(sizeof(S) == 8, "the other storages take their populations by bulk copies");
    constexpr int D = Lat<Q>::D;
    constexpr int HY = (D == 3) ? 1 : 0;  // halo rows along b
    constexpr int HW = TX + 2;
    constexpr int HH = TY + 2 * HY;
    constexpr int HN = HW * HH;
    constexpr int NT = TX * TY;
    constexpr int NBORDER = HN - NT;
    static_assert(D == 3 || TY == 1, "2-D tiles are one row");
    static_assert(NBORDER <= NT, "one border node per thread at most");

    T (*const sm)[3][HN] = reinterpret_cast<T(*)[3][HN]>(tlbm_smem);  // moment ring: rho, phi, psi over tile + halo

    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int A0 = w.A0, B0 = w.B0, M0 = w.M0, M1 = w.M1;
    const bool active = (A0 + tx < g.NA) && (B0 + ty < g.NB);

    // Node 0 of every thread: its own tile slot (coordinates wrap for threads past
    // the lattice edge, whose slots serve as the periodic halo of active ones).
    // Node 1: one border slot of the halo ring, for tid < NBORDER.
    int h[2], xc[2][3], yb[2][3];  // ring slot; byte offsets of x-1, x, x+1 in a row; rows b-1, b, b+1
    {
        int hx[2], hy[2];
        hx[0] = tx + 1;
        hy[0] = ty + HY;
        hx[1] = 0;
        hy[1] = 0;
        if (D == 2) {  // border nodes are summed by whole warps, below
            hx[1] = hx[0];
            hy[1] = hy[0];
        } else if (tid < HW) {
            hx[1] = tid;
        } else if (tid < 2 * HW) {
            hx[1] = tid - HW;
            hy[1] = HH - 1;
        } else if (tid < NBORDER) {
            const int k = tid - 2 * HW;
            hx[1] = k < HH - 2 ? 0 : HW - 1;
            hy[1] = 1 + (k < HH - 2 ? k : k - (HH - 2));
        } else {  // no border node: node 1 repeats node 0 (never used)
            hx[1] = hx[0];
            hy[1] = hy[0];
        }
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            h[n] = hy[n] * HW + hx[n];
            const int aa = modp(A0 + hx[n] - 1, g.NA);
            const int bb = (D == 3) ? modp(B0 + hy[n] - HY, g.NB) : 0;
            const int xs[3] = {wrap1(aa - 1, g.NA), aa, wrap1(aa + 1, g.NA)};
#pragma unroll
            for (int k = 0; k < 3; ++k) xc[n][k] = (xs[k] >> 5) * (int)Fmt<Q, S>::CHUNK + (xs[k] & 31) * Fmt<Q, S>::ESZ;
            yb[n][0] = (D == 3) ? wrap1(bb - 1, g.NB) : 0;
            yb[n][1] = bb;
            yb[n][2] = (D == 3) ? wrap1(bb + 1, g.NB) : 0;
        }
    }
    const int nnodes = D == 3 && tid < NBORDER ? 2 : 1;

    // D2Q9: the tile's two border nodes belong to warp 0 and warp 1 (both to the one
    // warp of a 32-node row).  Each of 27 lanes loads one of the node's populations
    // beside the loads of its own node; summed by one thread after its own node they
    // were a second load latency on every plane's path to the barrier.
    constexpr int BN = NT >= 64 ? 1 : 2;
    const int lane = tid & 31;
    const bool bwarp = D == 2 && (NT < 64 || tid < 64);
    int boff[BN], bslot[BN], bval_off = 0, bcm = 0;  // byte offset in a row, ring slot; of the lane's population
    if constexpr (D == 2) {
        const int l = lane < 3 * Q ? lane : 3 * Q - 1, bs = l / Q;
        int bca = 0;
        const int bdir = l % Q;
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (bdir == i && bs == c) {
                    bca = A::ca(i);
                    bcm = A::cm(i);
                    bval_off = Fmt<Q, S>::off(c, i);
                }
#pragma unroll
        for (int n = 0; n < BN; ++n) {
            const bool left = BN == 2 ? n == 0 : tid < 32;
            bslot[n] = left ? 0 : HW - 1;
            const int x = wrap1(modp(A0 + bslot[n] - 1, g.NA) - bca, g.NA);
            boff[n] = (x >> 5) * (int)Fmt<Q, S>::CHUNK + (x & 31) * Fmt<Q, S>::ESZ;
        }
    }

    const unsigned char* srcb = reinterpret_cast<const unsigned char*>(src);
    auto ldp = [&](const unsigned char* p, int s, int i) -> T { return Fmt<Q, S>::ld_delta(p, s, i); };
    // pull source of direction (ca, cb, cm) for node n at plane rows zr
    auto src_of = [&](int n, const int (&zr)[3], int ca, int cb, int cm) -> const unsigned char* {
        const long long row = (long long)zr[1 - cm] * g.NB + yb[n][1 - cb];
        return srcb + row * g.rowstride + xc[n][1 - ca];
    };

    // Phase M: moments of plane m for this thread's nodes into ring slot `slot`;
    // node 0's momentum density is returned in j and its rho in rd.
    auto moments_plane = [&](int m, int slot, T (&j)[3], T& rd) {
        const int mm = wrap1(m, g.NM);
        const int zr[3] = {wrap1(mm - 1, g.NM), mm, wrap1(mm + 1, g.NM)};
        const bool two = nnodes == 2;
        T rho0 = T(0), ja = T(0), jb = T(0), jm = T(0), phi0 = T(0), psi0 = T(0);
        T rho1 = T(0), phi1 = T(0), psi1 = T(0);
        T bval[BN];
        if constexpr (D == 2) {
            if (bwarp) {
                const int row = bcm == 0 ? zr[1] : (bcm > 0 ? zr[0] : zr[2]);
#pragma unroll
                for (int n = 0; n < BN; ++n)
                    bval[n] = *reinterpret_cast<const T*>(srcb + (long long)row * g.rowstride + boff[n] + bval_off);
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const unsigned char* p0 = src_of(0, zr, A::ca(i), A::cb(i), A::cm(i));
            const T f = ldp(p0, 0, i), gg = ldp(p0, 1, i), kk = ldp(p0, 2, i);
            rho0 += f;
            if (A::ca(i)) ja += T(A::ca(i)) * f;
            if (A::cb(i)) jb += T(A::cb(i)) * f;
            if (A::cm(i)) jm += T(A::cm(i)) * f;
            phi0 += gg;
            psi0 += kk;
        }
        if (two) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const unsigned char* p1 = src_of(1, zr, A::ca(i), A::cb(i), A::cm(i));
                rho1 += ldp(p1, 0, i);
                phi1 += ldp(p1, 1, i);
                psi1 += ldp(p1, 2, i);
            }
        }
        rd = rho0;
        sm[slot][0][h[0]] = rho0;
        sm[slot][1][h[0]] = phi0;
        sm[slot][2][h[0]] = psi0;
        if constexpr (D == 2) {
            if (bwarp) {
#pragma unroll
                for (int n = 0; n < BN; ++n) {  // lanes 0, 1, 2: rho, phi, psi in the order of the sums above
                    T acc = T(0);
#pragma unroll
                    for (int i = 0; i < Q; ++i) acc += __shfl_sync(0xffffffffu, bval[n], (lane % 3) * Q + i);
                    if (lane < 3) sm[slot][lane][bslot[n]] = acc;
                }
            }
        }
        if (two) {
            sm[slot][0][h[1]] = rho1;
            sm[slot][1][h[1]] = phi1;
            sm[slot][2][h[1]] = psi1;
        }
        j[0] = ja;
        j[1] = jb;
        j[2] = jm;
    };

    MassSum<T, false> msum;
    T jc[3], jn[3], rdc, rdn;

    grid_ready();
    moments_plane(M0 - 1, (M0 + 3) & 3, jn, rdn);
    moments_plane(M0, M0 & 3, jc, rdc);

    // derivatives: on D2Q9 the ring's planes go through the node's rolling sums in
    // order; on D3Q19 the 24 values they keep do not fit beside the collision in
    // 128 registers, and all three planes are read again (the same bits)
    constexpr bool KEEP = Q == 9;
    Roll<Q, T> roll;
    roll.clear();
    T X0[3], g12[3][3], l6[3];
    auto push_plane = [&](int m, T (&X)[3], T (&gr)[3][3], T (&la)[3]) {
        const int slot = m & 3;
        const T c1[3] = {sm[slot][0][h[0]], sm[slot][1][h[0]], sm[slot][2][h[0]]};
        roll.push([&](int k, int i, int jj) -> T { return sm[slot][k][h[0] + jj * HW + i]; }, c1, X, gr, la);
    };
    if (KEEP) {
        __syncthreads();
        push_plane(M0 + 3, X0, g12, l6);  // plane M0 - 1, in the slot of M0 + 3
        push_plane(M0, X0, g12, l6);
    }

    for (int m = M0; m < M1; ++m) {
        moments_plane(m + 1, (m + 1) & 3, jn, rdn);
        __syncthreads();
        if (!KEEP) {
            roll.clear();
            push_plane(m + 3, X0, g12, l6);  // plane m - 1
            push_plane(m, X0, g12, l6);
        }
        push_plane(m + 1, X0, g12, l6);
        if (active) {
            // the node's pulled populations: phase M read them one iteration ago
            const int zr[3] = {wrap1(m - 1, g.NM), m, wrap1(m + 1, g.NM)};
            T fv[Q], gv[Q], kv[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const unsigned char* pi = src_of(0, zr, A::ca(i), A::cb(i), A::cm(i));
                fv[i] = ldp(pi, 0, i);
                gv[i] = ldp(pi, 1, i);
                kv[i] = ldp(pi, 2, i);
            }
            const T jl[3] = {jc[0], D == 3 ? jc[1] : jc[2], D == 3 ? jc[2] : T(0)};  // lattice axes
            msum.add(rho_total<Q, S>(rdc), X0[1], X0[2]);
            unsigned char* out =
                reinterpret_cast<unsigned char*>(dst) + ((long long)m * g.NB + yb[0][1]) * g.rowstride + xc[0][1];
            collide_node<Q, S, false>(out, fv, gv, kv, rdc, X0, jl, g12, l6, P);
        }
        jc[0] = jn[0];
        jc[1] = jn[1];
        jc[2] = jn[2];
        rdc = rdn;
    }
    double mr, mp, ms;
    msum.get(mr, mp, ms);
    block_sum3(mr, mp, ms);
    if (tid == 0) put_block_sums(g, partials, bid, mr, mp, ms);
}

template <int Q, typename S, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, blocks_per_sm<S>(TX * TY))
k_fused(MGeom g, const S* __restrict__ src, S* __restrict__ dst, Phys<typename Store<S>::T> P,
        double* __restrict__ partials) {
    fused_body<Q, S, TX, TY>(g, src, dst, P, partials, blockIdx.x, work_of<TX, TY>(g, blockIdx.x));
}

// ------------------------------------------------------ solid-aware variant

// Bit i (1 <= i < Q) of nbm[r]: the pull source r - e_i of node r is solid;
// bit 0: r itself is solid.  Built once per lattice.
template <int Q>
__global__ void k_nbmask(Geom g, const uint8_t* __restrict__ solid, uint32_t* __restrict__ nbm) {
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
         r += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        coords(g, r, x, y, z);
        uint32_t m = solid[r] ? 1u : 0u;
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if (solid[node(g, wrap(x - Lat<Q>::cx(i), g.nx), wrap(y - Lat<Q>::cy(i), g.ny),
                           wrap(z - Lat<Q>::cz(i), g.nz))])
                m |= 1u << i;
        nbm[r] = m;
    }
}

// One step with solid nodes, halfway bounce-back and wetting ghosts.  As
// k_fused, but the ghost value of a solid node needs the moments of its fluid
// neighbours, so each block keeps a two-node halo and works two planes ahead:
//   M(m+2): moments of plane m+2 over tile + 2-node halo (solid nodes: 0)
//   barrier
//   G(m+1): ghost values of the solid nodes of plane m+1 over tile + 1-node halo
//           (mean over fluid axis neighbours of X - G_X; with only diagonal
//           fluid neighbours, of X - sqrt(2) G_X)
//   barrier
//   C(m):   derivatives, equilibria, BGK and store for the fluid tile nodes.
// The moment and mask rings have five plane slots and the momentum ring four, so
// a fast warp writing plane m+2 never touches data a slow warp still reads.
template <int Q, typename S>
__host__ __device__ constexpr int solid_smem(int TX, int TY) {
    const int hn = (TX + 4) * (TY + (Q == 19 ? 4 : 0)), t = (int)sizeof(typename Store<S>::T);
    return t * (15 * hn + 16 * TX * TY) + 4 * 5 * hn;
}

template <int Q, typename S, int TX, int TY, bool CHK = false>
__device__ __forceinline__ void solid_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                           const uint32_t* __restrict__ nbm,
                                           const Phys<typename Store<S>::T>& P, double* __restrict__ partials,
                                           const int bid, const Work w) {
    using T = typename Store<S>::T;
    using A = Axes<Q>;
    extern __shared__ __align__(16) unsigned char tlbm_smem[];
    constexpr int D = Lat<Q>::D;
    constexpr int H = 2;                  // halo width along a
    constexpr int HB = (D == 3) ? 2 : 0;  // halo width along b
    constexpr int HW = TX + 2 * H;
    constexpr int HH = TY + 2 * HB;
    constexpr int HN = HW * HH;
    constexpr int NT = TX * TY;
    constexpr int KS = (HN + NT - 1) / NT;  // region nodes per thread
    constexpr int R = 5;                    // plane slots of the rings
    static_assert(D == 3 || TY == 1, "2-D tiles are one row");
    static_assert(KS <= 3, "at most three region nodes per thread");

    // dynamic shared memory (solid_smem): effective rho, phi, psi (ghosts on solid
    // nodes), j and summed f deviations of the tile, neighbour masks
    T (*const sm)[3][HN] = reinterpret_cast<T(*)[3][HN]>(tlbm_smem);
    T (*const sj)[4][NT] = reinterpret_cast<T(*)[4][NT]>(tlbm_smem + sizeof(T) * R * 3 * HN);
    uint32_t (*const sk)[HN] = reinterpret_cast<uint32_t(*)[HN]>(tlbm_smem + sizeof(T) * (R * 3 * HN + 16 * NT));

    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int A0 = w.A0, B0 = w.B0, M0 = w.M0, M1 = w.M1;
    const bool active = (A0 + tx < g.NA) && (B0 + ty < g.NB);
    const long long plane = (long long)g.NA * g.NB;

    // this thread's region nodes h = tid + k NT: in-plane node index, pull-source
    // byte offsets along a and rows along b
    int xc[KS][3], yb[KS][3], rin[KS];
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const int h = min(tid + k * NT, HN - 1);
        const int hx = h % HW, hy = h / HW;
        const int aa = modp(A0 + hx - H, g.NA);
        const int bb = (D == 3) ? modp(B0 + hy - HB, g.NB) : 0;
        const int xs[3] = {wrap1(aa - 1, g.NA), aa, wrap1(aa + 1, g.NA)};
#pragma unroll
        for (int c = 0; c < 3; ++c) xc[k][c] = (xs[c] >> 5) * (int)Fmt<Q, S>::CHUNK + (xs[c] & 31) * Fmt<Q, S>::ESZ;
        yb[k][0] = (D == 3) ? wrap1(bb - 1, g.NB) : 0;
        yb[k][1] = bb;
        yb[k][2] = (D == 3) ? wrap1(bb + 1, g.NB) : 0;
        rin[k] = aa + g.NA * bb;
    }
    // the thread's own tile node (phase C): byte offsets of a-1, a, a+1, rows b-1, b, b+1
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
    const unsigned char* srcb = reinterpret_cast<const unsigned char*>(src);
    auto row_ptr = [&](int k, const int (&zr)[3], int cb, int cm) -> const unsigned char* {
        return srcb + ((long long)zr[1 - cm] * g.NB + yb[k][1 - cb]) * g.rowstride;
    };
    auto own_row = [&](const int (&zr)[3], int cb, int cm) -> const unsigned char* {
        return srcb + ((long long)zr[1 - cm] * g.NB + yo[1 - cb]) * g.rowstride;
    };

    // M: moments of plane m (node k's pulled populations, bounce-back at solids)
    auto moments_plane = [&](int m) {
        const int mm = modp(m, g.NM), slot = modp(m, R), js = modp(m, 4);
        const int zr[3] = {wrap1(mm - 1, g.NM), mm, wrap1(mm + 1, g.NM)};
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int h = tid + k * NT;
            if (h >= HN) break;
            const uint32_t mk = nbm[chk_index<CHK>(g, (long long)mm * plane + rin[k], plane * g.NM, 5)];
            T rd = T(0), ja = T(0), jb = T(0), jm = T(0), phi = T(0), psi = T(0);
            if (!(mk & 1u)) {
                const unsigned char* own = chk_node<Q, S, CHK>(g, srcb, row_ptr(k, zr, 0, 0) + xc[k][1], 2);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    // pull source, or this node's opposite run when the source is solid:
                    // one pointer select, then loads at the run offsets of direction i
                    // (pointer selects per set: f and g of a direction move together, k apart)
                    const unsigned char* p =
                        chk_node<Q, S, CHK>(g, srcb, row_ptr(k, zr, A::cb(i), A::cm(i)) + xc[k][1 - A::ca(i)], 1);
                    const bool bb = i > 0 && ((mk >> i) & 1u);
                    const unsigned char* pfg = bb ? own + (Fmt<Q, S>::off(0, opp<Q>(i)) - Fmt<Q, S>::off(0, i)) : p;
                    const unsigned char* pk = bb ? own + (Fmt<Q, S>::off(2, opp<Q>(i)) - Fmt<Q, S>::off(2, i)) : p;
                    T f, gv;
                    if (i > 0) Fmt<Q, S>::ld_fg(pfg, i, f, gv);
                    else f = Fmt<Q, S>::ld_delta(p, 0, 0), gv = Fmt<Q, S>::ld_delta(p, 1, 0);
                    rd += f;
                    if (A::ca(i)) ja += T(A::ca(i)) * f;
                    if (A::cb(i)) jb += T(A::cb(i)) * f;
                    if (A::cm(i)) jm += T(A::cm(i)) * f;
                    phi += gv;
                    psi += Fmt<Q, S>::ld_delta(pk, 2, i);
                }
            }
            const T rho = (mk & 1u) ? T(0) : (Fmt<Q, S>::OFFSET ? T(1) + rd : rd);
            sm[slot][0][h] = rho;
            sm[slot][1][h] = phi;
            sm[slot][2][h] = psi;
            sk[slot][h] = mk;
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

    // G: ghost values of the solid nodes of plane q within the one-node halo
    auto ghosts_plane = [&](int q) {
        const int slot = modp(q, R);
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int h = tid + k * NT;
            if (h >= HN) break;
            const int hx = h % HW, hy = h / HW;
            if (hx < 1 || hx > HW - 2 || (D == 3 && (hy < 1 || hy > HH - 2))) continue;
            const uint32_t mk = sk[slot][h];
            if (!(mk & 1u)) continue;
            T acc[3] = {T(0), T(0), T(0)};
            int n = 0;
#pragma unroll
            for (int i = 1; i <= Lat<Q>::NAXIS; ++i) {  // neighbour s + e_i is fluid?
                if ((mk >> opp<Q>(i)) & 1u) continue;
                const int sn = modp(q + A::cm(i), R);
                const int hn = (int)chk_index<CHK>(g, h + A::cb(i) * HW + A::ca(i), HN, 4);
#pragma unroll
                for (int c = 0; c < 3; ++c) acc[c] += sm[sn][c][hn] - P.Gw[c];
                ++n;
            }
            if (n == 0) {
                const T r2 = T(1.4142135623730951);
#pragma unroll
                for (int i = Lat<Q>::NAXIS + 1; i < Q; ++i) {
                    if ((mk >> opp<Q>(i)) & 1u) continue;
                    const int sn = modp(q + A::cm(i), R);
                    const int hn = (int)chk_index<CHK>(g, h + A::cb(i) * HW + A::ca(i), HN, 4);
#pragma unroll
                    for (int c = 0; c < 3; ++c) acc[c] += sm[sn][c][hn] - r2 * P.Gw[c];
                    ++n;
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) sm[slot][c][h] = n > 0 ? acc[c] / T(n) : T(0);
        }
    };

    constexpr bool PAIR = Fmt<Q, S>::OFFSET && !(Q == 19 && sizeof(S) == 4);
    constexpr bool HL = sizeof(S) == 4;  // evict-first hints in the collision
    MassSum<T, PAIR> msum;

    grid_ready();
    moments_plane(M0 - 2);
    moments_plane(M0 - 1);
    moments_plane(M0);
    moments_plane(M0 + 1);
    __syncthreads();
    ghosts_plane(M0 - 1);
    ghosts_plane(M0);
    __syncthreads();

    const int c0 = (ty + HB) * HW + tx + H;  // this thread's tile node in the region
    constexpr bool KEEP = Q == 9;  // as in fused_body
    Roll<Q, T> roll;
    roll.clear();
    auto push_plane = [&](int m, T (&X)[3], T (&gr)[3][3], T (&la)[3]) {
        const int slot = modp(m, R);
        const T c1[3] = {sm[slot][0][c0], sm[slot][1][c0], sm[slot][2][c0]};
        roll.push(
            [&](int k, int i, int jj) -> T {
                return sm[slot][k][(int)chk_index<CHK>(g, c0 + jj * HW + i, HN, 4)];
            },
            c1, X, gr, la);
    };
    if (KEEP) {
        T X0[3], g12[3][3], l6[3];
        push_plane(M0 - 1, X0, g12, l6);
        push_plane(M0, X0, g12, l6);
    }
    for (int m = M0; m < M1; ++m) {
        moments_plane(m + 2);
        __syncthreads();
        ghosts_plane(m + 1);
        __syncthreads();
        const uint32_t mk = sk[modp(m, R)][c0];
        T X0[3], g12[3][3], l6[3];
        if (!KEEP) {
            if (!active || (mk & 1u)) continue;
            roll.clear();
            push_plane(m - 1, X0, g12, l6);
            push_plane(m, X0, g12, l6);
        }
        push_plane(m + 1, X0, g12, l6);  // ghost values on solid neighbours
        if (KEEP && (!active || (mk & 1u))) continue;

        const int t = ty * TX + tx, js = modp(m, 4);
        const T jA = sj[js][0][t], jB = sj[js][1][t], jM = sj[js][2][t], rdc = sj[js][3][t];
        const T jl[3] = {jA, D == 3 ? jB : jM, D == 3 ? jM : T(0)};  // lattice axes
        if constexpr (PAIR) msum.add(rdc, X0[1], X0[2]);
        else msum.add(rho_total<Q, S>(rdc), X0[1], X0[2]);

        // ---- pulled populations (bounce-back at solid sources)
        const int zr[3] = {wrap1(m - 1, g.NM), m, wrap1(m + 1, g.NM)};
        const unsigned char* own = chk_node<Q, S, CHK>(g, srcb, own_row(zr, 0, 0) + xo[1], 2);
        T fv[Q], gv[Q], kv[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const unsigned char* p = chk_node<Q, S, CHK>(g, srcb, own_row(zr, A::cb(i), A::cm(i)) + xo[1 - A::ca(i)], 1);
            const bool bb = i > 0 && ((mk >> i) & 1u);
            const unsigned char* pfg = bb ? own + (Fmt<Q, S>::off(0, opp<Q>(i)) - Fmt<Q, S>::off(0, i)) : p;
            const unsigned char* pk = bb ? own + (Fmt<Q, S>::off(2, opp<Q>(i)) - Fmt<Q, S>::off(2, i)) : p;
            // the collision is the last reader of these lines: evict-first loads
            // (FP32 storage; measured slower for the 16-bit formats)
            if (i > 0) {
                Fmt<Q, S>::template ld_fg<HL>(pfg, i, fv[i], gv[i]);
            } else {
                fv[i] = HL ? Fmt<Q, S>::ld_last_delta(p, 0, 0) : Fmt<Q, S>::ld_delta(p, 0, 0);
                gv[i] = HL ? Fmt<Q, S>::ld_last_delta(p, 1, 0) : Fmt<Q, S>::ld_delta(p, 1, 0);
            }
            kv[i] = HL ? Fmt<Q, S>::ld_last_delta(pk, 2, i) : Fmt<Q, S>::ld_delta(pk, 2, i);
        }

        // ---- collide + store
        unsigned char* out = chk_node<Q, S, CHK>(
            g, reinterpret_cast<unsigned char*>(dst),
            reinterpret_cast<unsigned char*>(dst) + ((long long)m * g.NB + yo[1]) * g.rowstride + xo[1], 3);
        // streamed out (evict-first, FP32): read only by the next step
        collide_node<Q, S, HL>(out, fv, gv, kv, rdc, X0, jl, g12, l6, P);
    }

    double mr, mp, ms;
    msum.get(mr, mp, ms);
    block_sum3(mr, mp, ms);
    if (tid == 0) put_block_sums(g, partials, bid, mr, mp, ms);
}

// BPS, blocks per SM: D3Q19 in FP32 and 16 bits spills at 128 registers (FP32 296 bytes
// a thread).  Alone on the lattice three blocks with 168 are faster (5 % solid nodes,
// FP32: 128^3 468 us a step with four, 416 with three; 40^3 47.5 and 36.8); beside the
// clean blocks' launch four are (144x128x80, drop on a wall: 50 steps 10.99 and 11.53 ms).
template <int Q, typename S, int TX, int TY, bool CHK = false, int BPS = blocks_per_sm<S>(TX * TY)>
__global__ void __launch_bounds__(TX * TY, BPS)
k_fused_solid(MGeom g, const S* __restrict__ src, S* __restrict__ dst, const uint32_t* __restrict__ nbm,
              Phys<typename Store<S>::T> P, double* __restrict__ partials) {
    solid_body<Q, S, TX, TY, CHK>(g, src, dst, nbm, P, partials, blockIdx.x, work_of<TX, TY>(g, blockIdx.x));
}

// ------------------------------------------------------------- batches

// One member of a batched step: its geometry, buffers for this step's parity,
// neighbour mask (solid lattices), physics, partial sums and first block.
template <typename T>
struct SimDesc {
    MGeom g;
    const void* src;
    void* dst;
    const uint32_t* nbm;
    Phys<T> P;
    double* partials;
    double* step_mass;
    int* flag;
    int block0;  // first block of this member in the batched grid
    int nblocks;
};

// block -> member: the last descriptor whose block0 <= blockIdx.x; the member's
// descriptor is copied to shared memory for the body to read
template <typename T>
__device__ __forceinline__ const SimDesc<T>& batch_member(const SimDesc<T>* __restrict__ d, int nsims,
                                                          SimDesc<T>& sh) {
    if (threadIdx.x == 0) {
        int lo = 0, hi = nsims - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (d[mid].block0 <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        sh = d[lo];
    }
    __syncthreads();
    return sh;
}

// p, known to point to global memory: pointers read from a descriptor are generic to
// the compiler, whose generic loads and stores may alias the shared rings and run
// one after another (16 lattices of 768x384, FP32: 330 us a step against 176 of one
// lattice of their size)
template <typename P>
__device__ __forceinline__ P* as_global(P* p) {
    __builtin_assume(__isGlobal(p));
    return p;
}
// a member's geometry in registers: the descriptor in shared memory could alias the
// rings as well
__device__ __forceinline__ MGeom member_geom(const MGeom& m) {
    MGeom g = m;
    if (g.items) g.items = as_global(g.items);
    g.flag = as_global(g.flag);
    return g;
}

// FP64 totals of every member: block i sums member i's partials in a fixed order
template <typename T>
__global__ void k_mass_final_batch(const SimDesc<T>* __restrict__ d) {
    const SimDesc<T>& m = d[blockIdx.x];
    double a = 0.0, b = 0.0, c = 0.0;
    for (int k = threadIdx.x; k < m.nblocks; k += blockDim.x) {
        a += m.partials[3 * k];
        b += m.partials[3 * k + 1];
        c += m.partials[3 * k + 2];
    }
    block_sum3(a, b, c);
    if (threadIdx.x == 0) {
        m.step_mass[0] = a;
        m.step_mass[1] = b;
        m.step_mass[2] = c;
        if (!(isfinite(a) && isfinite(b) && isfinite(c))) atomicOr(m.flag, 1);
    }
}

}  // namespace tlbm_dev
