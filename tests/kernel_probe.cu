// kernel_probe.cu -- the marching kernels with bulk copies, launched on geometries that
// the engine never gives them: test_gpu_kernel_probe.py.  Every buffer is larger than
// anything a launch here can reach.
#include <vector>

#include "../paper_1511_02155_gb300/csrc/tlbm_launch.cuh"

using namespace tlbm_dev;

namespace {

struct Lattice {
    MGeom g{};
    unsigned char *src = nullptr, *dst = nullptr;
    double* partials = nullptr;
    int* flag = nullptr;
    unsigned long long* check = nullptr;
    Phys<float> P{};
    ~Lattice() {
        cudaFree(src);
        cudaFree(dst);
        cudaFree(partials);
        cudaFree(flag);
        cudaFree(check);
        cudaFree(const_cast<int4*>(g.items));
    }
    template <int Q>
    cudaError_t make(int nx, int ny, int nz, int TX, int TY) {
        const int ncx = (nx + 31) / 32;
        g.NA = nx;
        g.NB = Q == 19 ? ny : 1;
        g.NM = Q == 19 ? nz : ny;
        g.rowstride = (long long)ncx * Fmt<Q, float>::CHUNK;
        g.NC = 1;
        g.bytes = (long long)g.NB * g.NM * g.rowstride;
        g.tilesA = (nx + TX - 1) / TX;
        g.tilesB = (g.NB + TY - 1) / TY;
        for (int m = 0; m < 3; ++m) P.kappa[m] = 0.01f, P.omega[m] = 1.0f;
        P.a2 = P.gamma[0] = P.gamma[1] = 1.0f;
        cudaError_t e = cudaMalloc(&src, g.bytes);
        if (e == cudaSuccess) e = cudaMalloc(&dst, g.bytes);
        if (e == cudaSuccess) e = cudaMalloc(&partials, 3 * sizeof(double) * 64);
        if (e == cudaSuccess) e = cudaMalloc(&flag, sizeof(int));
        if (e == cudaSuccess) e = cudaMalloc(&check, sizeof(unsigned long long));
        if (e == cudaSuccess) e = cudaMemset(src, 0, g.bytes);
        if (e == cudaSuccess) e = cudaMemset(dst, 0xab, g.bytes);
        if (e == cudaSuccess) e = cudaMemset(flag, 0, sizeof(int));
        if (e == cudaSuccess) e = cudaMemset(check, 0, sizeof(unsigned long long));
        g.flag = flag;
        g.check = check;
        return e;
    }
    // bytes of dst that a launch has changed
    cudaError_t changed(long long* n) {
        std::vector<unsigned char> h((size_t)g.bytes);
        const cudaError_t e = cudaMemcpy(h.data(), dst, h.size(), cudaMemcpyDeviceToHost);
        *n = 0;
        for (unsigned char b : h) *n += b != 0xab;
        return e;
    }
};

}  // namespace

// A step whose waits run out: blocks of fewer threads than their barriers count.  The
// flag that they raise, the bytes of the new state that they stored, and the seconds.
extern "C" int probe_late(int Q, int* flag, long long* stored, double* seconds) {
    Lattice l;
    cudaError_t e;
    if (Q == 19) e = l.make<19>(40, 9, 6, 32, 4);
    else e = l.make<9>(200, 12, 1, 128, 1);
    cudaEvent_t a = nullptr, b = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    if (e == cudaSuccess) e = cudaEventRecord(a);
    const float* src = reinterpret_cast<const float*>(l.src);
    float* dst = reinterpret_cast<float*>(l.dst);
    const int nb = l.g.tilesA * l.g.tilesB;
    if (e == cudaSuccess) {
        if (Q == 19)  // 96 of 128: the fourth row's warp is missing
            e = launch_smem(k_bulk<float, false>, BulkShape<float>::SMEM, 96, 2, nb, nullptr, l.g, src, dst, l.P, l.partials);
        else  // 32 of 128: the thread that expects the bulk copies is missing
            e = launch_smem(k_bulk2<float, 128, false>, Bulk2Shape<float, 128>::SMEM, 32, 4, nb, nullptr, l.g, src, dst, l.P,
                            l.partials);
    }
    if (e == cudaSuccess) e = cudaEventRecord(b);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    if (e == cudaSuccess) e = cudaMemcpy(flag, l.flag, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = l.changed(stored);
    *seconds = ms * 1e-3;
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    return (int)e;
}

// The checked step of planes M0 .. M1 - 1 of one tile, told that the populations end
// `cut` bytes before they do: the word that it records.
extern "C" int probe_check(int Q, int M0, int M1, long long cut, unsigned long long* word, long long* bytes) {
    Lattice l;
    cudaError_t e;
    if (Q == 19) e = l.make<19>(40, 9, 8, 32, 4);
    else e = l.make<9>(200, 8, 1, 128, 1);
    l.g.bytes -= cut;
    *bytes = l.g.bytes;
    int4* items = nullptr;
    const int4 it = make_int4(0, 0, M0, 2 * M1);
    if (e == cudaSuccess) e = cudaMalloc(&items, sizeof it);
    l.g.items = items;
    if (e == cudaSuccess) e = cudaMemcpy(items, &it, sizeof it, cudaMemcpyHostToDevice);
    const float* src = reinterpret_cast<const float*>(l.src);
    float* dst = reinterpret_cast<float*>(l.dst);
    if (e == cudaSuccess) {
        if (Q == 19) e = launch_bulk<float>(k_bulk<float, true>, 1, nullptr, l.g, src, dst, l.P, l.partials);
        else e = launch_bulk2<float, 128>(k_bulk2<float, 128, true>, 1, nullptr, l.g, src, dst, l.P, l.partials);
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(word, l.check, sizeof *word, cudaMemcpyDeviceToHost);
    return (int)e;
}
