// host_rules.cu -- the marching step's dispatch rules (tlbm_launch.cuh) without a
// device: test_host_rules.py.
#include "../paper_1511_02155_gb300/csrc/tlbm_launch.cuh"

// blocks of one step of a lattice, or -1 where the step refuses it
template <int Q, typename S>
static long long blocks(tlbm_host::DevState& d) {
    std::vector<int4> items;
    std::vector<uint8_t> units;
    if (d.solid) {  // a wall of solid nodes on the first plane
        units.assign((size_t)d.ny * d.nz * d.ncx, 0);
        std::fill(units.begin(), units.begin() + (Q == 9 ? 1 : d.ny) * d.ncx, (uint8_t)3);
        d.units = units.data();
        d.ndirty = tlbm_dev::solid_items<Q, S>(d, items);
        d.nitems = (int)items.size();
        d.items = items.data();
    }
    const long long nb = tlbm_dev::fused_blocks<Q, S>(d);
    return nb > 0x7fffffffLL || nb > d.partials_cap ? -1 : nb;
}

extern "C" long long rule_blocks(int Q, int prec, int nx, int ny, int nz, int solid, int coupling, int tile, int sms) {
    tlbm_host::DevState d{};
    static const uint8_t some = 1;
    d.Q = Q;
    d.prec = prec;
    d.nx = nx;
    d.ny = ny;
    d.nz = nz;
    d.N = (long long)nx * ny * nz;
    d.ncx = (nx + 31) / 32;
    d.solid = solid ? &some : nullptr;
    d.coupling = coupling;
    d.tile = tile;
    d.sms = sms;
    d.partials_cap = std::max(d.N / 64 + 1, (long long)tlbm_host::kMassBlocks);
    if (Q == 9) return prec == 0 ? blocks<9, double>(d) : blocks<9, float>(d);
    return prec == 0 ? blocks<19, double>(d) : blocks<19, float>(d);
}

// longest block of planes near solid nodes on a D2Q9 FP32 lattice that has them
// everywhere but in `clean` planes of its last 32-node column
extern "C" int rule_longest_dirty(int nx, int ny, int clean, int sms) {
    tlbm_host::DevState d{};
    static const uint8_t some = 1;
    d.Q = 9;
    d.prec = 1;
    d.nx = nx;
    d.ny = ny;
    d.nz = 1;
    d.N = (long long)nx * ny;
    d.ncx = (nx + 31) / 32;
    d.solid = &some;
    d.sms = sms;
    d.partials_cap = std::max(d.N / 64 + 1, (long long)tlbm_host::kMassBlocks);
    std::vector<uint8_t> units((size_t)ny * d.ncx, (uint8_t)1);
    for (int m = 0; m < clean; ++m) units[(size_t)(ny / 2 + m) * d.ncx + d.ncx - 1] = 0;
    d.units = units.data();
    std::vector<int4> items;
    const int dirty = tlbm_dev::solid_items<9, float>(d, items);
    int most = 0;
    for (int k = 0; k < dirty; ++k) most = std::max(most, (items[k].w >> 1) - items[k].z);
    return most;
}
