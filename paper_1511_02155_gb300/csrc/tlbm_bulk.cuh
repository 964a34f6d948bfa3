// tlbm_bulk.cuh -- the periodic D3Q19 and D2Q9 steps with their populations brought
// into shared memory by bulk copies (FP32 and 16-bit storage; Semprebon, Krueger,
// Kusumaatmaja, arXiv:1511.02155), and the kernels that mix these with the
// solid-aware step (k_mix) or run many lattices in one launch (k_*_batch).
//
// The marching scheme is that of tlbm_fused.cuh: a block owns one 32-node chunk of
// x by TY rows and marches along z; the moments of a plane over the tile and its
// one-node halo go to a shared ring, and the plane before it is collided with the
// derivatives they complete.  What bounds that scheme with ordinary loads is the
// latency of some 80 loads a node at 16 warps per SM (registers) and the L1 that
// holds them in flight.  Here no thread waits for a load: while a plane is worked
// on, the next one is copied by the TMA unit.  The layout makes that cheap: all
// populations that a row of nodes pulls from one source row (y - e_y, z - e_z) are
// one contiguous piece of a chunk, so nine copies of 384 or 1152 bytes (FP32) bring
// a row's 57 populations, already in the place where the pull wants them but for
// the x shift, which is a lane offset in shared memory.  The x neighbours beyond
// the chunk are 114 single words per row, copied by 4- and 8-byte cp.async.
//
// Per plane p of a block's M1 - M0 + 2:
//   wait for the copies of p
//   populations of p into registers, moments of p: own node and at most one border
//   node per thread -> ring
//   barrier: nothing of the slot is needed any more
//   start the copies of p + 1 into it
//   derivatives of p - 1 (Roll), collision of p - 1 from registers, store
// One slot: the copies run while the plane before is collided, the larger part of
// the work, and the other blocks of the SM fill what wait is left.  A second slot
// measured slower (side by side, with 4-byte words at the ends: FP32 1.96 against 1.55
// ms at 256^3, FP16 1.38 against 1.00; the present kernel takes 1.46 to 1.54 and 1.04): it
// takes the L1 that the words of x neighbours need on their way, a 128-byte line
// for each.  One barrier a plane, since the ring holds two planes or more.
#pragma once

#include "tlbm_fused.cuh"

namespace tlbm_dev {

// What a row of nodes pulls, as runs of 32 lane words in shared memory.  FP32: the
// chunk's own order.  16-bit formats: the chunk's first 26 runs, then the k words
// whose two directions come from different rows, once for each direction.
template <typename S, int Q = 19>
struct RowImage {
    using F = Fmt<Q, S>;
    static constexpr bool PACKED = F::PACKED;
    static constexpr int KEPT = Q == 19 ? 26 : 14;  // 16-bit: runs of one source row each
    static constexpr int RUNS = PACKED ? (Q == 19 ? 34 : 16) : 3 * Q;
    static constexpr int BYTES = RUNS * 128;
    static constexpr int COPIES = PACKED ? (Q == 19 ? 17 : 5) : (Q == 19 ? 9 : 3);
    // byte offset of (s, i)
    __host__ __device__ static constexpr int off(int s, int i) {
        if (PACKED && s == 2 && i > 0 && F::krun(i) >= KEPT) return krun2(i) * 128 + F::khalf(i) * 2;
        return F::off(s, i);
    }
    __host__ __device__ static constexpr int krun2(int i) {  // D3Q19 3 4 5 6 11 14 12 13, D2Q9 3 4
        if (Q == 9) return 11 + i;
        return i <= 6 ? 23 + i : (i == 11 ? 30 : (i == 14 ? 31 : (i == 12 ? 32 : 33)));
    }
    // copy n: (e_y, e_z) of its source row, offset in the chunk and in the image, bytes
    struct Copy {
        int ey, ez, src, dst, bytes;
    };
    __host__ __device__ static constexpr Copy copy(int n) {
        if (Q == 9) {  // groups e_y = 0, 1, -1, then the k word of 3 and of 4
            const int len0 = PACKED ? 6 : 9, len = PACKED ? 4 : 9, e = n == 0 ? 0 : (n == 1 || n == 3 ? 1 : -1);
            const int at = n == 0 ? 0 : (n <= 2 ? len0 + (n - 1) * len : KEPT);
            return Copy{e, 0, at * 128, (n <= 2 ? at : KEPT + n - 3) * 128, (n == 0 ? len0 : (n <= 2 ? len : 1)) * 128};
        }
        constexpr int ey[9] = {0, 1, -1, 0, 0, 1, 1, -1, -1}, ez[9] = {0, 0, 0, 1, -1, 1, -1, 1, -1};
        if (n >= 9) {  // 16-bit: a k word for one of its two directions
            constexpr int d[8] = {3, 4, 5, 6, 11, 14, 12, 13};
            const int i = d[n < 17 ? n - 9 : 0];
            return Copy{Lat<Q>::cy(i), Lat<Q>::cz(i), F::krun(i) * 128, krun2(i) * 128, 128};
        }
        // runs before group n and in it
        const int len0 = PACKED ? 6 : 9, len = PACKED ? 4 : 9, one = PACKED ? 1 : 3;
        const int at = n == 0 ? 0 : (n <= 4 ? len0 + (n - 1) * len : len0 + 4 * len + (n - 5) * one);
        const int runs = n == 0 ? len0 : (n <= 4 ? len : one);
        return Copy{ey[n], ez[n], at * 128, at * 128, runs * 128};
    }
    static __device__ __forceinline__ float value(const unsigned char* n, int s, int i) {
        if constexpr (PACKED) {
            if (i > 0) return Store<S>::get(*reinterpret_cast<const S*>(n + off(s, i)));
        }
        return *reinterpret_cast<const float*>(n + off(s, i));
    }
    // populations of direction i
    static __device__ __forceinline__ void load(const unsigned char* n, int i, float& f, float& g, float& k) {
        if constexpr (PACKED) {
            if (i > 0) {
                Store<S>::get2(*reinterpret_cast<const unsigned*>(n + off(0, i)), f, g);
                k = value(n, 2, i);
                return;
            }
        }
        f = value(n, 0, i);
        g = value(n, 1, i);
        k = value(n, 2, i);
    }
};

// A node's populations in registers: as FP32 values, except for D3Q19 in 16 bits,
// where they keep their stored form (39 registers instead of 57; converted where
// they are used).
template <typename S, int Q = 19>
struct NodePops {
    using I = RowImage<S, Q>;
    static constexpr bool STORED = I::PACKED && Q == 19;
    float f[Q], g[Q], k[Q];  // values (STORED: of the rest populations)
    unsigned fg[Q];          // STORED: (f, g) words, k
    unsigned short kh[Q];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            f[i] = g[i] = k[i] = 0.0f;
            fg[i] = 0u;
            kh[i] = 0;
        }
    }
    // take direction i from the slot, and return its values
    __device__ __forceinline__ void take(const unsigned char* n, int i, float& f_, float& g_, float& k_) {
        if (STORED && i > 0) {
            fg[i] = *reinterpret_cast<const unsigned*>(n + I::off(0, i));
            kh[i] = *reinterpret_cast<const unsigned short*>(n + I::off(2, i));
        } else {
            I::load(n, i, f[i], g[i], k[i]);
        }
        get(i, f_, g_, k_);
    }
    __device__ __forceinline__ void get(int i, float& f_, float& g_, float& k_) const {
        if constexpr (STORED) {
            if (i > 0) {
                Store<S>::get2(fg[i], f_, g_);
                k_ = Store<S>::get(*reinterpret_cast<const S*>(&kh[i]));
                return;
            }
        }
        f_ = f[i];
        g_ = g[i];
        k_ = k[i];
    }
};

// ------------------------------------------------------------- PTX wrappers

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase with this parity, for at most about a second: false then.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
    if (mbar_try(bar, parity)) return true;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
#pragma unroll 1
        for (int n = 0; n < 64; ++n)
            if (mbar_try(bar, parity)) return true;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    } while (t - t0 < 1000000000ull);
    return false;
}
// A thread whose wait has run out is late for the rest of its march: it stores nothing
// more, starts no copy and does not arrive, so that the phases it should arrive at stay
// open and the block's other threads run out of their next wait in turn.  It gives the
// copies in flight a second wait before it goes on, so that the block's shared memory
// is not given up under them.  (Each thread's own words, not a vote at the barrier:
// __syncthreads_or cost 1 % of a step on 517x391 in 16 bits.)
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void copy4(unsigned dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy8(unsigned dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
// this thread's cp.async so far arrive at the barrier when they are done
__device__ __forceinline__ void copy_arrive(unsigned bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// ------------------------------------------------------------------ kernel

template <typename S>
struct BulkShape {
    static constexpr int TY = 4;                                 // rows of a tile
    static constexpr bool FRESH = RowImage<S>::PACKED;           // derivatives from three ring planes
    static constexpr int ROWS = TY + 2;                          // tile and halo rows
    static constexpr int SIDE = ROWS * RowImage<S>::BYTES;       // x neighbours, in the lanes of one more row
    static constexpr int SLOT = SIDE + RowImage<S>::BYTES;
    static constexpr int THREADS = 32 * TY;
    static constexpr int RN = ROWS * 34;                         // a ring plane: tile and halo
    static constexpr int NRING = FRESH ? 4 : 2;                  // planes of the ring
    static constexpr int RING = SLOT, BAR = RING + NRING * 3 * RN * 4;
    static constexpr int SMEM = BAR + 16;
    static constexpr int BPS = RowImage<S>::PACKED ? 3 : 2;      // blocks per SM, by shared memory and registers
    static_assert(ROWS * 4 <= 32 && BAR % 8 == 0, "side lanes; barrier alignment");
    static_assert(ROWS * RowImage<S>::COPIES <= THREADS, "one bulk copy per thread");
};

template <typename S, bool CHK>
__device__ __forceinline__ void bulk_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                          const Phys<float>& P, double* __restrict__ partials, const int bid) {
    constexpr int Q = 19;
    using F = Fmt<Q, S>;
    using I = RowImage<S>;
    using B = BulkShape<S>;
    using L = Lat<Q>;
    constexpr int TY = B::TY;
    extern __shared__ __align__(128) unsigned char tlbm_bulk_smem[];
    float* const ring = reinterpret_cast<float*>(tlbm_bulk_smem + B::RING);
    const unsigned char* const sl = tlbm_bulk_smem;
    const unsigned smem0 = smem_u32(tlbm_bulk_smem), bar = smem0 + B::BAR;

    const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
    const Work wk = work_of<32, TY>(g, bid);
    const int chunk = wk.A0 >> 5, B0 = wk.B0, M0 = wk.M0, M1 = wk.M1;
    const int W = min(32, g.NA - 32 * chunk);  // nodes of this chunk
    const int H = min(TY, g.NB - B0);          // rows of this tile
    const int rows = H + 2;
    bool active = lane < W && ty < H;
    const unsigned char* const srcb = reinterpret_cast<const unsigned char*>(src);
    const long long pstride = (long long)g.NB * g.rowstride;
    const int last = M1 - M0 + 1;  // planes 0 .. last of the march: M0 - 1 .. M1

    // ---- this thread's bulk copy: row, group and source row are fixed
    const unsigned char* bsrc = srcb;
    unsigned bdst = 0, bbytes = 0;
    int bez = 0;
    if (tid < rows * I::COPIES) {
        const int r = tid / I::COPIES, n = tid % I::COPIES;
        typename I::Copy c = I::copy(0);
#pragma unroll
        for (int k = 1; k < I::COPIES; ++k) {
            const typename I::Copy ck = I::copy(k);
            if (n == k) c = ck;
        }
        const int y = modp(B0 + r - 1 - c.ey, g.NB);
        bsrc = chk_node<Q, S, CHK>(g, srcb, srcb + y * g.rowstride + chunk * F::CHUNK, 1) + c.src;
        bdst = (unsigned)chk_index<CHK>(g, r * I::BYTES + c.dst, B::SIDE - c.bytes + 1, 4);
        bbytes = c.bytes;
        bez = c.ez;
    }
    // ---- this thread's x neighbours: (row, direction) items, two to three lane words
    // each of one position (e_x = 0, either side) or of two adjacent ones (e_x != 0).
    // Lane 4 r + {0, 1, 2, 3} of the side row holds x0 - 2, x0 - 1, x0 + W, x0 + W + 1
    // of row r.
    constexpr int NPOS = 28;  // 9 directions with e_x = 0, twice; 10 others
    constexpr int NI = (B::ROWS * NPOS + B::THREADS - 1) / B::THREADS;
    const unsigned char* isrc[NI];
    unsigned idst[NI], idel[NI];  // image offset; deltas of the second word: chunk << 16 | image
    int iez[NI];                  // e_z, + 8 where a third word follows, + 16 for two positions
    int idx2[NI];                 // bytes to the second position's word: 4 where one 8-byte copy serves
#pragma unroll
    for (int k = 0; k < NI; ++k) {
        const int it = tid + k * B::THREADS;
        isrc[k] = nullptr;
        idst[k] = idel[k] = 0;
        iez[k] = idx2[k] = 0;
        if (it < rows * NPOS) {
            const int r = it / NPOS, p = it % NPOS;
            const int slot = p < 18 ? 1 + (p & 1) : (p < 23 ? 0 : 2);
            const int mu = slot < 2 ? slot - 2 : W + slot - 2;
            const int which = p < 18 ? p / 2 : (p < 23 ? p - 18 : p - 23);
            int o0 = 0, o1 = 0, d0 = 0, d1 = 0, ey = 0, ez = 0;
            int n0 = 0, np = 0, nm = 0;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const bool mine = L::cx(i) == 0 ? (p < 18 && which == n0)
                                                : (L::cx(i) > 0 ? (p >= 18 && p < 23 && which == np) : (p >= 23 && which == nm));
                if (mine) {
                    o0 = F::off(0, i);
                    d0 = I::off(0, i);
                    // second word: 16-bit the k word, else (and for the rest) g, and then k
                    o1 = (I::PACKED && i > 0) ? F::krun(i) * 128 : F::off(1, i);
                    d1 = (I::PACKED && i > 0) ? I::off(2, i) - F::khalf(i) * 2 : I::off(1, i);
                    ey = L::cy(i);
                    ez = L::cz(i) + ((I::PACKED && i > 0) ? 0 : 8);
                }
                n0 += L::cx(i) == 0;
                np += L::cx(i) > 0;
                nm += L::cx(i) < 0;
            }
            const int x = modp(32 * chunk + mu, g.NA), x2 = modp(x + 1, g.NA), y = modp(B0 + r - 1 - ey, g.NB);
            const int at = (x >> 5) * (int)F::CHUNK + (x & 31) * 4, at2 = (x2 >> 5) * (int)F::CHUNK + (x2 & 31) * 4;
            isrc[k] = chk_node<Q, S, CHK>(g, srcb, srcb + y * g.rowstride + at, 1) + o0;
            idst[k] = (unsigned)chk_index<CHK>(g, B::SIDE + d0 + (4 * r + slot) * 4, B::SLOT - 4, 4);
            idel[k] = (unsigned)(o1 - o0) << 16 | (unsigned)(d1 - d0);
            // two positions: one 8-byte copy where both lanes are one aligned pair
            idx2[k] = (at2 - at == 4 && (x & 1) == 0) ? 4 : at2 - at + 1;
            iez[k] = ez + (p < 18 ? 0 : 16);
        }
    }
    // byte offsets of the planes z - 1, z, z + 1 of the march plane whose copies start next
    long long zm = (long long)modp(M0 - 2, g.NM) * pstride, zc = (long long)modp(M0 - 1, g.NM) * pstride,
              zp = (long long)modp(M0, g.NM) * pstride;
    const long long zend = (long long)g.NM * pstride;
    auto start = [&]() {
        if (tid == 0) mbar_expect(bar, rows * I::BYTES);
        if (bbytes)
            bulk_load(smem0 + bdst, chk_span<CHK>(g, srcb, bsrc + (bez == 0 ? zc : (bez > 0 ? zm : zp)), bbytes, 1), bbytes,
                      bar);
#pragma unroll
        for (int k = 0; k < NI; ++k) {
            if (isrc[k]) {
                const bool two = iez[k] >= 15, third = ((iez[k] + 1) & 8) != 0;  // e_z + 8 third + 16 two
                const int ez = ((iez[k] + 1) & 7) - 1;
                const unsigned char* s = isrc[k] + (ez == 0 ? zc : (ez > 0 ? zm : zp));
                const unsigned d = smem0 + idst[k], dd = idel[k] & 0xffffu, ds = idel[k] >> 16;
                auto c4 = [&](unsigned to, const unsigned char* from) { copy4(to, chk_span<CHK>(g, srcb, from, 4, 1)); };
                auto c8 = [&](unsigned to, const unsigned char* from) { copy8(to, chk_span<CHK>(g, srcb, from, 8, 1)); };
                if (two && idx2[k] == 4) {
                    c8(d, s);
                    c8(d + dd, s + ds);
                    if (third) c8(d + 2 * dd, s + 2 * ds);
                } else {
                    c4(d, s);
                    c4(d + dd, s + ds);
                    if (third) c4(d + 2 * dd, s + 2 * ds);
                    if (two) {
                        const unsigned char* s2 = s + (idx2[k] - 1);
                        c4(d + 4, s2);
                        c4(d + 4 + dd, s2 + ds);
                        if (third) c4(d + 4 + 2 * dd, s2 + 2 * ds);
                    }
                }
            }
        }
        copy_arrive(bar);
        zm = zc;
        zc = zp;
        zp = zp + pstride == zend ? 0 : zp + pstride;
    };

    if (tid == 0) {
        mbar_init(bar, B::THREADS + 1);  // every thread's cp.async, and the bulk copies' bytes
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    grid_ready();
    start();

    // ---- offsets in a slot of the words that a node at lane mu of row r pulls, for
    // e_x = 0, +1 (from mu - 1), -1 (from mu + 1)
    auto word = [&](int r, int mu) -> int {
        const int at = mu >= 0 && mu < W ? r * I::BYTES + mu * 4
                                         : B::SIDE + (4 * r + (mu < 0 ? mu + 2 : min(mu - W, 1) + 2)) * 4;
        return (int)chk_index<CHK>(g, at, B::SIDE + 128, 4);  // its last run ends in the slot
    };
    const int r0 = ty + 1;
    const int own[3] = {r0 * I::BYTES + lane * 4, word(r0, lane - 1), word(r0, lane + 1)};
    const int c0 = r0 * 34 + lane + 1;  // own node in the ring
    // border node: rows 0 and H + 1 over W + 2 columns, then the two side columns
    int bord[3] = {0, 0, 0}, cb = -1;
    if (tid < 2 * (W + 2) + 2 * H) {
        int r, q;
        if (tid < 2 * (W + 2)) {
            r = tid < W + 2 ? 0 : H + 1;
            q = tid < W + 2 ? tid : tid - (W + 2);
        } else {
            const int k = tid - 2 * (W + 2);
            r = 1 + (k >> 1);
            q = (k & 1) ? W + 1 : 0;
        }
        bord[0] = word(r, q - 1);
        bord[1] = word(r, q - 2);
        bord[2] = word(r, q);
        cb = (int)chk_index<CHK>(g, r * 34 + q, B::RN, 4);
    }
    unsigned char* const outb =
        reinterpret_cast<unsigned char*>(dst) + (active ? (long long)(B0 + ty) * g.rowstride : 0) +
        (long long)chunk * F::CHUNK + lane * F::ESZ;

    MassSum<float, I::PACKED> msum;
    Roll<Q, float> roll;
    roll.clear();
    NodePops<S> cur, nxt;
    cur.clear();
    float jc[3] = {0.0f, 0.0f, 0.0f}, rdc = 0.0f;
    int upto = last;  // copies of the planes up to here; below 0: late

#pragma unroll 1
    for (int p = 0; p <= last; ++p) {
        if (upto >= 0 && !mbar_wait(bar, p & 1)) {
            upto = -1;
            active = false;
            mbar_wait(bar, p & 1);
        }

        // ---- populations and moments of plane p
        float* const rg = ring + (p & (B::NRING - 1)) * 3 * B::RN;
        float jn[3] = {0.0f, 0.0f, 0.0f}, rdn = 0.0f, c1[3] = {0.0f, 0.0f, 0.0f};
        {
            const unsigned char* const b0 = sl + own[0];
            const unsigned char* const bp = sl + own[1];
            const unsigned char* const bm = sl + own[2];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const unsigned char* n = L::cx(i) == 0 ? b0 : (L::cx(i) > 0 ? bp : bm);
                float f, gg, kk;
                nxt.take(n, i, f, gg, kk);
                rdn += f;
                if (L::cx(i)) jn[0] += (float)L::cx(i) * f;
                if (L::cy(i)) jn[1] += (float)L::cy(i) * f;
                if (L::cz(i)) jn[2] += (float)L::cz(i) * f;
                c1[1] += gg;
                c1[2] += kk;
            }
            c1[0] = rdn + 1.0f;
            if (active) {
                rg[c0] = c1[0];
                rg[B::RN + c0] = c1[1];
                rg[2 * B::RN + c0] = c1[2];
            }
        }
        if (cb >= 0) {
            const unsigned char* const b0 = sl + bord[0];
            const unsigned char* const bp = sl + bord[1];
            const unsigned char* const bm = sl + bord[2];
            float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const unsigned char* n = L::cx(i) == 0 ? b0 : (L::cx(i) > 0 ? bp : bm);
                float f, gg, kk;
                I::load(n, i, f, gg, kk);
                s0 += f;
                s1 += gg;
                s2 += kk;
            }
            rg[cb] = s0 + 1.0f;
            rg[B::RN + cb] = s1;
            rg[2 * B::RN + cb] = s2;
        }
        __syncthreads();  // the slot is read, the ring written
        if (p < upto) start();

        // ---- derivatives and collision of plane p - 1
        if (active) {
            float X[3], g12[3][3], l6[3];
            auto push = [&](const float* const rq, const float (&c)[3]) {
                roll.push(
                    [&](int k, int i, int jj) -> float {
                        return rq[k * B::RN + (int)chk_index<CHK>(g, c0 + jj * 34 + i, B::RN, 4)];
                    },
                    c, X, g12, l6);
            };
            if (B::FRESH) {
                roll.clear();
#pragma unroll
                for (int k = 2; k >= 1; --k) {
                    const float* const rq = ring + ((p - k) & (B::NRING - 1)) * 3 * B::RN;
                    const float c[3] = {rq[c0], rq[B::RN + c0], rq[2 * B::RN + c0]};
                    push(rq, c);
                }
            }
            push(rg, c1);
            if (p >= 2) {
                if constexpr (I::PACKED) msum.add(rdc, X[1], X[2]);
                else msum.add(rho_total<Q, S>(rdc), X[1], X[2]);
                unsigned char* const out = chk_node<Q, S, CHK>(g, reinterpret_cast<unsigned char*>(dst),
                                                               outb + (long long)(M0 + p - 2) * pstride, 3);
                float fv[Q], gv[Q], kv[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) cur.get(i, fv[i], gv[i], kv[i]);
                collide_node<Q, S, true>(out, fv, gv, kv, rdc, X, jc, g12, l6, P);
            }
        }
        cur = nxt;
        jc[0] = jn[0];
        jc[1] = jn[1];
        jc[2] = jn[2];
        rdc = rdn;
    }
    if (upto < 0) atomicOr(g.flag, 2);  // a copy did not arrive: the step's results are void
    double mr, mp, ms;
    msum.get(mr, mp, ms);
    block_sum3(mr, mp, ms);
    if (tid == 0) put_block_sums(g, partials, bid, mr, mp, ms);
}

// ---------------------------------------------------------------- D2Q9

// The same for D2Q9 (periodic body of FP32 and 16-bit storage): a block owns TX nodes of
// a row, TX / 32 chunks with three copies each (five in 16 bits), and marches along y.
// Only the two words beyond either end of the tile come by cp.async.  The kernel it
// replaces loaded a plane's 27 populations a node, summed, waited at the barrier
// and only then collided: at 16 warps an SM its waits filled 60 % of the time.  Two
// slots of 17 kB (FP32, TX 128) leave room for four blocks an SM; the copies of
// p + 2 start at p's barrier.  The two border nodes go to three lanes each of the last
// two warps, one set of populations a lane.  A step of whole passes before and
// after: FP32 512x256 12.0 and 11.0 us, 1000x701 46 and 36, 4096x4096 720 and 696;
// kernel alone, FP16 1000x701 41 and 24, 2048x1024 84 and 55, 4096x4096 498 and 406.
// FP16 517x391 is slower, 15.1 and 16.1: four planes a block, and the copies of the
// first two hidden by nothing.
template <typename S, int TX>
struct Bulk2Shape {
    using I = RowImage<S, 9>;
    static constexpr int CH = TX / 32;
    static constexpr int SIDE = CH * I::BYTES;       // x neighbours: lanes 0..3 of one more chunk image
    static constexpr int SLOT = SIDE + I::BYTES;
    static constexpr int RN = TX + 2;
    static constexpr int RING = 2 * SLOT, BAR = (RING + 2 * 3 * RN * 4 + 7) / 8 * 8;
    static constexpr int SMEM = BAR + 16;
    static constexpr int ITEMS = 18;                 // (direction, x neighbour) pairs
};

template <typename S, int TX, bool CHK>
__device__ __forceinline__ void bulk2_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                           const Phys<float>& P, double* __restrict__ partials, const int bid,
                                           const Work wk) {
    constexpr int Q = 9;
    using F = Fmt<Q, S>;
    using I = RowImage<S, Q>;
    using B = Bulk2Shape<S, TX>;
    using L = Lat<Q>;
    extern __shared__ __align__(16) unsigned char tlbm_smem[];
    float* const ring = reinterpret_cast<float*>(tlbm_smem + B::RING);
    const unsigned smem0 = smem_u32(tlbm_smem), bar0 = smem0 + B::BAR;

    const int tid = threadIdx.x;
    const int A0 = wk.A0, M0 = wk.M0, M1 = wk.M1;
    const int W = min(TX, g.NA - A0);  // nodes of this tile
    bool active = tid < W;
    const unsigned char* const srcb = reinterpret_cast<const unsigned char*>(src);
    const int last = M1 - M0 + 1;

    // ---- this thread's bulk copy (threads of the second warp)
    const unsigned char* bsrc = srcb;
    unsigned bdst = 0, bbytes = 0;
    int bey = 0;
    const int nch = (W + 31) >> 5;
    {
        const int t = tid - 32;
        if (t >= 0 && t < nch * I::COPIES) {
            const int c = t / I::COPIES, n = t % I::COPIES;
            typename I::Copy cp = I::copy(0);
#pragma unroll
            for (int k = 1; k < I::COPIES; ++k) {
                const typename I::Copy ck = I::copy(k);
                if (n == k) cp = ck;
            }
            bsrc = chk_node<Q, S, CHK>(g, srcb, srcb + (A0 / 32 + c) * F::CHUNK, 1) + cp.src;
            bdst = (unsigned)chk_index<CHK>(g, c * I::BYTES + cp.dst, B::SIDE - cp.bytes + 1, 4);
            bbytes = cp.bytes;
            bey = cp.ey;
        }
    }
    // ---- this thread's x neighbour (threads 0 .. 17): lanes {0, 1, 2, 3} of the side
    // image hold A0 - 2, A0 - 1, A0 + W, A0 + W + 1; directions with e_x = 0 need the
    // inner two, e_x = 1 the left two, e_x = -1 the right two
    const unsigned char* isrc = srcb;
    unsigned idst = 0, idel_s = 0, idel_d = 0;
    int iey = 0;
    bool ithird = false;
    if (tid < B::ITEMS) {
        const int p = tid, which = p < 6 ? p / 2 : (p - 6) % 6 / 2;
        const int slot = p < 6 ? 1 + (p & 1) : (p < 12 ? (p & 1) : 2 + (p & 1));
        const int mu = slot < 2 ? slot - 2 : W + slot - 2;
        int o0 = 0, o1 = 0, d0 = 0, d1 = 0, n0 = 0, np = 0, nm = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const bool mine = L::cx(i) == 0 ? (p < 6 && which == n0)
                                            : (L::cx(i) > 0 ? (p >= 6 && p < 12 && which == np) : (p >= 12 && which == nm));
            if (mine) {
                o0 = F::off(0, i);
                d0 = I::off(0, i);
                o1 = (I::PACKED && i > 0) ? F::krun(i) * 128 : F::off(1, i);
                d1 = (I::PACKED && i > 0) ? I::off(2, i) - F::khalf(i) * 2 : I::off(1, i);
                iey = L::cy(i);
                ithird = !(I::PACKED && i > 0);
            }
            n0 += L::cx(i) == 0;
            np += L::cx(i) > 0;
            nm += L::cx(i) < 0;
        }
        const int x = modp(A0 + mu, g.NA);
        isrc = chk_node<Q, S, CHK>(g, srcb, srcb + (x >> 5) * F::CHUNK + (x & 31) * F::ESZ, 1) + o0;
        idst = (unsigned)chk_index<CHK>(g, B::SIDE + d0 + slot * 4, B::SLOT - 4, 4);
        idel_s = (unsigned)(o1 - o0);
        idel_d = (unsigned)(d1 - d0);
    }
    // byte offsets of the rows y - 1, y, y + 1 of the plane whose copies start next
    long long ym = (long long)modp(M0 - 2, g.NM) * g.rowstride, yc = (long long)modp(M0 - 1, g.NM) * g.rowstride,
              yp = (long long)modp(M0, g.NM) * g.rowstride;
    const long long yend = (long long)g.NM * g.rowstride;
    auto start = [&](int p) {
        const unsigned sl = smem0 + (p & 1) * B::SLOT, bar = bar0 + (p & 1) * 8;
        if (tid == 32) mbar_expect(bar, nch * I::BYTES);
        if (bbytes)
            bulk_load(sl + bdst, chk_span<CHK>(g, srcb, bsrc + (bey == 0 ? yc : (bey > 0 ? ym : yp)), bbytes, 1), bbytes, bar);
        if (tid < B::ITEMS) {
            const unsigned char* s = isrc + (iey == 0 ? yc : (iey > 0 ? ym : yp));
            const unsigned d = sl + idst;
            auto c4 = [&](unsigned to, const unsigned char* from) { copy4(to, chk_span<CHK>(g, srcb, from, 4, 1)); };
            c4(d, s);
            c4(d + idel_d, s + idel_s);
            if (ithird) c4(d + 2 * idel_d, s + 2 * idel_s);
            copy_arrive(bar);
        }
        ym = yc;
        yc = yp;
        yp = yp + g.rowstride == yend ? 0 : yp + g.rowstride;
    };
    if (tid == 0) {
        mbar_init(bar0, B::ITEMS + 1);
        mbar_init(bar0 + 8, B::ITEMS + 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    grid_ready();
    start(0);
    start(1);

    // offset in a slot of the lane word of tile node x (-2 .. W + 1)
    auto word = [&](int x) -> int {
        const int at = x >= 0 && x < W ? (x >> 5) * I::BYTES + (x & 31) * 4
                                       : B::SIDE + (x < 0 ? x + 2 : min(x - W, 1) + 2) * 4;
        return (int)chk_index<CHK>(g, at, B::SIDE + 128, 4);  // its last run ends in the slot
    };
    const int own[3] = {(tid >> 5) * I::BYTES + (tid & 31) * 4, word(tid - 1), word(tid + 1)};
    // the two border nodes: lanes 0, 1, 2 of the last two warps, one set each
    const int bx = tid < TX - 32 ? -1 : W, bset = tid & 31;
    const bool border = tid >= TX - 64 && bset < 3;
    const int bord[3] = {word(bx), word(bx - 1), word(bx + 1)};
    unsigned char* const outb = reinterpret_cast<unsigned char*>(dst) +
                                (active ? (long long)((A0 + tid) >> 5) * F::CHUNK : 0) + (tid & 31) * F::ESZ;

    MassSum<float, true> msum;
    Roll<Q, float> roll;
    roll.clear();
    NodePops<S, Q> cur, nxt;
    cur.clear();
    float jc[3] = {0.0f, 0.0f, 0.0f}, rdc = 0.0f;
    int upto = last;  // as in bulk_body
#pragma unroll 1
    for (int p = 0; p <= last; ++p) {
        if (upto >= 0 && !mbar_wait(bar0 + (p & 1) * 8, (p >> 1) & 1)) {
            upto = -1;
            active = false;
            mbar_wait(bar0 + (p & 1) * 8, (p >> 1) & 1);
            if (p < last) mbar_wait(bar0 + ((p + 1) & 1) * 8, ((p + 1) >> 1) & 1);
        }

        // ---- populations and moments of plane p
        const unsigned char* const sl = tlbm_smem + (p & 1) * B::SLOT;
        float* const rg = ring + (p & 1) * 3 * B::RN + 1;  // rg[0]: tile node 0
        float jn[3] = {0.0f, 0.0f, 0.0f}, rdn = 0.0f, c1[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float f, gg, kk;
            nxt.take(sl + own[L::cx(i) == 0 ? 0 : (L::cx(i) > 0 ? 1 : 2)], i, f, gg, kk);
            rdn += f;
            if (L::cx(i)) jn[0] += (float)L::cx(i) * f;
            if (L::cy(i)) jn[1] += (float)L::cy(i) * f;
            c1[1] += gg;
            c1[2] += kk;
        }
        c1[0] = rdn + 1.0f;
        if (active) {
            rg[tid] = c1[0];
            rg[B::RN + tid] = c1[1];
            rg[2 * B::RN + tid] = c1[2];
        }
        if (border) {  // in the order of the sums above
            float acc = 0.0f;
            if (!I::PACKED || bset < 2) {
                const int so = bset * 128, sh = I::PACKED ? bset * 2 : so;  // from f to g, k: runs; 16-bit: halves
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const unsigned char* n = sl + bord[L::cx(i) == 0 ? 0 : (L::cx(i) > 0 ? 1 : 2)] + I::off(0, i);
                    if (I::PACKED && i > 0) acc += Store<S>::get(*reinterpret_cast<const S*>(n + sh));
                    else acc += *reinterpret_cast<const float*>(n + so);
                }
            } else {
#pragma unroll
                for (int i = 0; i < Q; ++i) acc += I::value(sl + bord[L::cx(i) == 0 ? 0 : (L::cx(i) > 0 ? 1 : 2)], 2, i);
            }
            rg[bset * B::RN + bx] = bset == 0 ? acc + 1.0f : acc;
        }
        __syncthreads();  // the slot is read, the ring written
        if (p + 2 <= upto) start(p + 2);

        // ---- derivatives and collision of plane p - 1
        if (active) {
            float X[3], g12[3][3], l6[3];
            roll.push(
                [&](int k, int i, int) -> float {
                    return rg[k * B::RN + (int)chk_index<CHK>(g, tid + i + 1, B::RN, 4) - 1];
                },
                c1, X, g12, l6);
            if (p >= 2) {
                msum.add(rdc, X[1], X[2]);
                unsigned char* const out = chk_node<Q, S, CHK>(g, reinterpret_cast<unsigned char*>(dst),
                                                               outb + (long long)(M0 + p - 2) * g.rowstride, 3);
                float fv[Q], gv[Q], kv[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) cur.get(i, fv[i], gv[i], kv[i]);
                collide_node<Q, S, true>(out, fv, gv, kv, rdc, X, jc, g12, l6, P);
            }
        }
        cur = nxt;
        jc[0] = jn[0];
        jc[1] = jn[1];
        rdc = rdn;
    }
    if (upto < 0) atomicOr(g.flag, 2);  // a copy did not arrive: the step's results are void
    double mr, mp, ms;
    msum.get(mr, mp, ms);
    block_sum3(mr, mp, ms);
    if (tid == 0) put_block_sums(g, partials, bid, mr, mp, ms);
}

template <typename S, int TX, bool CHK>
__global__ void __launch_bounds__(TX, 512 / TX)
k_bulk2(MGeom g, const S* __restrict__ src, S* __restrict__ dst, Phys<float> P, double* __restrict__ partials) {
    bulk2_body<S, TX, CHK>(g, src, dst, P, partials, blockIdx.x, work_of<TX, 1>(g, blockIdx.x));
}

template <typename S, bool CHK>
__global__ void __launch_bounds__(BulkShape<S>::THREADS, BulkShape<S>::BPS)
k_bulk(MGeom g, const S* __restrict__ src, S* __restrict__ dst, Phys<float> P, double* __restrict__ partials) {
    bulk_body<S, CHK>(g, src, dst, P, partials, blockIdx.x);
}

template <typename S>
__global__ void __launch_bounds__(BulkShape<S>::THREADS, BulkShape<S>::BPS)
k_bulk_batch(const SimDesc<float>* __restrict__ d, int nsims) {
    __shared__ SimDesc<float> sh;
    const SimDesc<float>& m = batch_member(d, nsims, sh);
    bulk_body<S, false>(member_geom(m.g), as_global(static_cast<const S*>(m.src)), as_global(static_cast<S*>(m.dst)),
                        m.P, as_global(m.partials), (int)blockIdx.x - m.block0);
}

// ------------------------------------------------- solid lattices, batches

// D2Q9 with solid nodes: a block whose planes keep two nodes away from every solid
// node runs the periodic body, the others the solid-aware one (which blocks is
// decided per lattice, Work).  The solid-aware body costs twice as much: two
// barriers a plane, four halo planes, two loads of every mask.  FP32 4096x2048 with 32 wells
// (2.6 % of its planes near solids): 502 us a step by the solid-aware body alone, 290
// mixed.
template <int Q, typename S>
struct Mix {
    static constexpr bool DBL = sizeof(S) == 8;
    template <int TX>
    static constexpr int smem() {
        int a = 0;
        if constexpr (DBL) a = fused_smem<Q, S>(TX, 1);
        else a = Bulk2Shape<S, TX>::SMEM;
        return a > solid_smem<Q, S>(TX, 1) ? a : solid_smem<Q, S>(TX, 1);
    }
};
template <int Q, typename S, int TX, bool CHK = false>
__device__ __forceinline__ void mix_body(const MGeom& g, const S* __restrict__ src, S* __restrict__ dst,
                                         const uint32_t* __restrict__ nbm, const Phys<typename Store<S>::T>& P,
                                         double* __restrict__ partials, const int bid) {
    const Work w = work_of<TX, 1>(g, bid);
    if (w.dirty) solid_body<Q, S, TX, 1, CHK>(g, src, dst, nbm, P, partials, bid, w);
    else if constexpr (sizeof(S) == 8) fused_body<Q, S, TX, 1>(g, src, dst, P, partials, bid, w);
    else bulk2_body<S, TX, CHK>(g, src, dst, P, partials, bid, w);
}
template <int Q, typename S, int TX, bool CHK = false>
__global__ void __launch_bounds__(TX, blocks_per_sm<S>(TX))
k_mix(MGeom g, const S* __restrict__ src, S* __restrict__ dst, const uint32_t* __restrict__ nbm,
      Phys<typename Store<S>::T> P, double* __restrict__ partials) {
    mix_body<Q, S, TX, CHK>(g, src, dst, nbm, P, partials, blockIdx.x);
}

template <int Q, typename S, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, blocks_per_sm<S>(TX * TY))
k_fused_batch(const SimDesc<typename Store<S>::T>* __restrict__ d, int nsims) {
    __shared__ SimDesc<typename Store<S>::T> sh;
    const SimDesc<typename Store<S>::T>& m = batch_member(d, nsims, sh);
    const int bid = (int)blockIdx.x - m.block0;
    const MGeom g = member_geom(m.g);
    const S* src = as_global(static_cast<const S*>(m.src));
    S* dst = as_global(static_cast<S*>(m.dst));
    double* partials = as_global(m.partials);
    const Work w = work_of<TX, TY>(g, bid);
    if constexpr (sizeof(S) == 8) fused_body<Q, S, TX, TY>(g, src, dst, m.P, partials, bid, w);
    else bulk2_body<S, TX, false>(g, src, dst, m.P, partials, bid, w);
}

template <int Q, typename S, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, blocks_per_sm<S>(TX * TY))
k_fused_solid_batch(const SimDesc<typename Store<S>::T>* __restrict__ d, int nsims) {
    __shared__ SimDesc<typename Store<S>::T> sh;
    const SimDesc<typename Store<S>::T>& m = batch_member(d, nsims, sh);
    const int bid = (int)blockIdx.x - m.block0;
    const S* src = as_global(static_cast<const S*>(m.src));
    S* dst = as_global(static_cast<S*>(m.dst));
    const uint32_t* nbm = as_global(m.nbm);
    double* partials = as_global(m.partials);
    const MGeom g = member_geom(m.g);
    if constexpr (Q == 9) mix_body<Q, S, TX>(g, src, dst, nbm, m.P, partials, bid);
    else solid_body<Q, S, TX, TY>(g, src, dst, nbm, m.P, partials, bid, work_of<TX, TY>(g, bid));
}

}  // namespace tlbm_dev
