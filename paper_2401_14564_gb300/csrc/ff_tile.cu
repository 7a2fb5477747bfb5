// K1 by tiles: force-field grid assembly (Sec. 5.1.1 step 1) with the far atoms of each 16x16x16-node tile
// summed at its interpolation points (ff_tile.cuh says how and how exactly); the sums, options and outputs
// are those of ff_assemble.cu, whose direct kernel remains for samples of a few atoms and for the split
// grids.  Tiles start at multiples of 16 nodes whatever layers a call asks for, and a node's value depends on
// its tile alone, so layer ranges, launch shapes and the batch write the same bits.
#include "ff_tile.cuh"


namespace pp {
namespace {

// Grids of fewer tiles than CTAs fit the GPU (two per SM), or of a few more, which a second wave of a few tiles ends,
// run by halves: 48 tiles of a 40-atom molecule 27 -> 18 us, 196 of a 120-atom periodic sheet 144 -> 115 us, 308 of 67
// atoms 53 -> 39, 324 of 492 atoms 361 -> 297; with more tiles the far sums made twice cost more than the better
// balance gives (490 tiles of 407 atoms 109 -> 154, 780 of an 80-atom molecule 60 -> 79 us).  By quarters no grid ran faster.
constexpr int kHalfFifths = 11;  // 2.2 tiles per SM

// kEnergy: E alone, one float per node (tricubic grids).  kForcesOnly: E slots written as 0.
// kParts: CTAs to a tile (1 or 2), which share its layers (all sum the far atoms).  A tile over a molecule has
// every atom near and takes several times one beside it; a grid of few tiles ends with it.
// kThin: for layer ranges that start or end inside a half tile (256x256 nodes, 4 layers of the 60-atom flake 20.5 -> 16.6 us,
// of an 800-atom periodic sheet on 300x300 216 -> 168; direct sums 16.4 and 219; across a tile's edge 27 and 269).
template <bool kMinImage, bool kCutoff, bool kQuad, bool kEnergy, bool kForcesOnly, int kParts, bool kThin>
__global__ void __launch_bounds__(kTileThreads, 2) ff_tile_kernel(const FFLaunch P) {
    __shared__ TileShared S;
    const TileJob J = {P.x, P.y, P.z, P.R, P.eps, P.q, P.n, P.x0, P.y0, P.z0, P.dx, P.dy, P.dz, P.map.nx, P.map.ny};
    const FFConst c = ff_const(P.R_pp, P.eps_pp, P.kQ, P.core_frac, P.Lx, P.Ly, kCutoff ? P.coul_rc : 0.f,
                               kQuad ? P.kQzz : 0.f);
    const int z = kParts == 2 ? blockIdx.z >> 1 : blockIdx.z, only = kParts == 2 ? blockIdx.z & 1 : -1;
    const int k0 = (P.kbeg / kTileN + z) * kTileN;
    if (kParts == 2 && (k0 + 8 * only >= P.kend || k0 + 8 * only + 8 <= P.kbeg)) return;
    ff_tile<kMinImage, kCutoff, kQuad, kEnergy, kForcesOnly, kThin>(
        J, c, blockIdx.x * kTileN, blockIdx.y * kTileN, k0, S,
        [&](int f, int n) { return (kParts == 1 || f >> 3 == only) && k0 + f < P.kend && k0 + f + n > P.kbeg; },
        [&](int i, int j, int k, float2 fx, float2 fy, float2 fz, float2 en) {
            if (i >= P.map.nx || j >= P.map.ny) return;
            const int base_xy = axis_off(P.map.ax, i) + axis_off(P.map.ay, j);
            auto at = [&](int kk) { return checked(base_xy + axis_off(P.map.az, kk), P.map.stored_nodes, kChkGridWrite); };
            const bool w0 = k >= P.kbeg && k < P.kend, w1 = k + 1 >= P.kbeg && k + 1 < P.kend;
            if constexpr (kEnergy) {
                if (w0) P.ffE[at(k)] = en.x;
                if (w1) P.ffE[at(k + 1)] = en.y;
            } else {
                if (kForcesOnly) en = make_float2(0.f, 0.f);
                if (w0) P.ff[at(k)] = make_float4(fx.x, fy.x, fz.x, en.x);
                if (w1) P.ff[at(k + 1)] = make_float4(fx.y, fy.y, fz.y, en.y);
            }
        });
}

}  // namespace

cudaError_t launch_ff_tiles(const FFLaunch& L, cudaStream_t s) {
    dim3 grid((L.map.nx + kTileN - 1) / kTileN, (L.map.ny + kTileN - 1) / kTileN,
              (L.kend + kTileN - 1) / kTileN - L.kbeg / kTileN);
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t tiles = (int64_t)grid.x * grid.y * grid.z;
    const int parts = 5 * tiles < (int64_t)kHalfFifths * sms ? 2 : 1;
    grid.z *= parts;
    const bool thin = L.kbeg % 8 != 0 || (L.kend % 8 != 0 && L.kend != L.map.nz);
    with_flags(L.min_image != 0, L.coul_rc > 0.f, L.kQzz != 0.f, [&](auto mi, auto cut, auto quad) {
        constexpr bool MI = decltype(mi)::value, CUT = decltype(cut)::value, QUAD = decltype(quad)::value;
        auto go = [&](auto energy, auto forces) {
            constexpr bool E = decltype(energy)::value, F = decltype(forces)::value;
            auto run = [&](auto k) { k<<<grid, kTileThreads, 0, s>>>(L); };
            if (parts == 2) thin ? run(ff_tile_kernel<MI, CUT, QUAD, E, F, 2, true>) : run(ff_tile_kernel<MI, CUT, QUAD, E, F, 2, false>);
            else thin ? run(ff_tile_kernel<MI, CUT, QUAD, E, F, 1, true>) : run(ff_tile_kernel<MI, CUT, QUAD, E, F, 1, false>);
        };
        if (L.map.interp == 1) go(std::true_type{}, std::false_type{});
        else if (L.forces_only) go(std::false_type{}, std::true_type{});
        else go(std::false_type{}, std::false_type{});
        return 0;
    });
    return cudaGetLastError();
}

PP_CHECK_READER(check_flags_ff_tile)

}  // namespace pp
