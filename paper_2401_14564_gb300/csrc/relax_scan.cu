// K2: relaxed tip scan (Sec. 5.1.1 step 2) with an optional fused df epilogue.
//
// One thread owns one pixel column and walks its heights from the top down:
// the PP starts at anchor + d0 for the first height and at p*(k-1) - dz z_hat
// (the tip moved down by dz, the deflection kept) for the others, and is
// relaxed by FIRE on G(p) = F_T(p) + F_S(p) (Eq. F_PP), with the tip springs
// of Eq. F_tip and F_S trilinearly interpolated from the force grid.  The tip
// force is read out as Fz = -F^T_{R,z} = kR (|d| - R0) d_z / |d| (Sec. 2.1).
//
// The FIRE state is e = d - d0, the deflection from the spring's rest
// displacement.  Then |d|^2 - R0^2 = (2 d0 + e).e + (|d0|^2 - R0^2) is formed
// without cancellation, so the radial extension and Fz keep full FP32
// relative precision however stiff the spring (with d itself the extension
// would be quantised at ulp(R0) ~ 5e-7 A, i.e. 3e-4 eV/A at 1e4 N/m).
//
// Lanes of a warp cover an 8x4 pixel tile (a smaller one in scans too small to
// fill the GPU, see tile_shape), so the 32 PPs sit in neighbouring
// grid cells and their corner loads share L1 lines.  Each lane advances to its
// next height as soon as it has converged; the warp only waits for its
// slowest lane once, at the end of the columns, not at every height.
// Interpolation is done by hand in FP32 from eight float4 corner loads on the
// read-only path (hardware texture filtering carries only 8 fractional bits
// in its weights, which would cost the 1e-3 A position parity).
#include "relax_core.cuh"

namespace pp {
namespace {

constexpr int kThreads = 32;  // one warp per CTA: one pixel tile (evens out warps per SM)

// Node range [lo, hi] (clamped to the grid) covering coordinates a..b along one axis.
__device__ __forceinline__ int2 node_range(float a, float b, float inv_d, float g0s, int n) {
    const float fa = fmaf(fminf(a, b), inv_d, g0s), fb = fmaf(fmaxf(a, b), inv_d, g0s);
    const int lo = min(max(__float2int_rd(fa), 0), n - 1);
    const int hi = min(max(__float2int_rd(fb) + 1, 0), n - 1);
    return make_int2(lo, hi);
}

// Linear layout: ask L2 for the grid rows under this warp's tile over the
// z-range its PPs will visit (anchor heights + d0, 0.5 A margin), so that the
// scan's first touches of the slab are served in parallel at the start instead
// of one demand miss at a time inside the FIRE loops.  Rows are contiguous in
// x; each lane issues a bulk prefetch (a hint: it never faults and changes no
// result) for every 32nd row.  Lateral deflections reach the neighbouring
// tiles' rows, which those warps prefetch.
template <bool kNarrow>
__device__ __forceinline__ void prefetch_tile_slab(const RelaxLaunch& P, int tx, int ty, int lane) {
    const int wsh = kNarrow ? P.tile_wsh : 3, hsh = kNarrow ? P.tile_hsh : 2;
    const int ia = tx << wsh, ib = min(ia + (1 << wsh), P.snx) - 1;
    const int ja = ty << hsh, jb = min(ja + (1 << hsh), P.sny) - 1;
    const int2 ri = node_range(fmaf((float)ia, P.spx, P.sx0) + P.d0x, fmaf((float)ib, P.spx, P.sx0) + P.d0x,
                               P.inv_dx, P.gx0s, P.map.nx);
    const int2 rj = node_range(fmaf((float)ja, P.spy, P.sy0) + P.d0y, fmaf((float)jb, P.spy, P.sy0) + P.d0y,
                               P.inv_dy, P.gy0s, P.map.ny);
    const float ztop = P.z_top + P.d0z, zbot = P.z_top - (P.snz - 1) * P.sdz + P.d0z;
    const int2 rk = node_range(fminf(ztop, zbot) - 0.5f, fmaxf(ztop, zbot) + 0.5f, P.inv_dz, P.gz0s, P.map.nz);
    const int nj = rj.y - rj.x + 1, rows = nj * (rk.y - rk.x + 1);
    for (int r = lane; r < rows; r += kThreads) {
        const int j = rj.x + r % nj, k = rk.x + r / nj;
        const int first = node_index(P.map, ri.x, j, k);
        if (P.map.interp == 0) {
            const unsigned bytes = (unsigned)(ri.y - ri.x + 1) * 16u;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.ff + first), "r"(bytes) : "memory");
        } else {
            // one float per node: the whole 16-byte groups inside the row (one node wider
            // on the left for the tricubic stencil); up to 3 nodes at the right end are left out
            const int lo = max(first - 1, 0) & ~3, hi = (first + (ri.y - ri.x) + 1) & ~3;
            if (hi > lo)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.ffE + lo), "r"((unsigned)(hi - lo) * 4u)
                             : "memory");
        }
    }
}

// The warp's lowest and highest node layer read, folded into P.zspan by lane 0 (all 32 lanes call).
__device__ __forceinline__ void record_zspan(const RelaxLaunch& P, int2 span) {
    const int lo = __reduce_min_sync(0xffffffffu, span.x);
    const int hi = __reduce_max_sync(0xffffffffu, span.y);
    if (threadIdx.x == 0) {
        atomicMin(P.zspan, lo);
        atomicMax(P.zspan + 1, hi);
    }
}

// Lane l's pixel of tile (tx, ty), x fastest inside the tile; idle past its pixels.
template <bool kNarrow>
__device__ __forceinline__ void tile_pixel(const RelaxLaunch& P, int tx, int ty, int& i, int& j) {
    const int wsh = kNarrow ? P.tile_wsh : 3, hsh = kNarrow ? P.tile_hsh : 2;
    const int lane = threadIdx.x, dj = lane >> wsh;
    i = (tx << wsh) + (lane & ((1 << wsh) - 1));
    j = (ty << hsh) + dj;
    if (kNarrow && (dj >> hsh)) i = P.snx;
}

// This warp's pixel (i, j); i = snx marks an idle lane.  Without a plan: lane l of the tile
// (blockIdx.x, blockIdx.y), lanes past the tile's pixels idle.  With one (a 1-D grid): the first
// plan_hblocks warps take the plan's listed pixels, plan_lanes lanes each (-1 or anything outside the
// scan: idle), and warp plan_hblocks + t takes tile t less the listed pixels.  *tx < 0: no tile (no
// slab prefetch).
template <bool kNarrow>
__device__ __forceinline__ void scan_pixel(const RelaxLaunch& P, int& i, int& j, int& tx, int& ty) {
    const int lane = threadIdx.x;
    if (!P.plan_list) {
        tx = blockIdx.x;
        ty = blockIdx.y;
        tile_pixel<kNarrow>(P, tx, ty, i, j);
        return;
    }
    const int npix = P.snx * P.sny;
    const int b = blockIdx.x;
    if (b < P.plan_hblocks) {
        tx = ty = -1;
        int p = -1;
        if (lane < P.plan_lanes) p = P.plan_list[b * P.plan_lanes + lane];
        const bool ok = p >= 0 && p < npix;
        i = ok ? p % P.snx : P.snx;
        j = ok ? p / P.snx : P.sny;
        return;
    }
    const int wsh = kNarrow ? P.tile_wsh : 3;
    const int ntx = (P.snx + (1 << wsh) - 1) >> wsh, t = b - P.plan_hblocks;
    tx = t % ntx;
    ty = t / ntx;
    tile_pixel<kNarrow>(P, tx, ty, i, j);
    if (i < P.snx && j < P.sny) {
        const int p = j * P.snx + i;
        if ((P.plan_mask[p >> 5] >> (p & 31)) & 1u) i = P.snx;  // run by a plan warp
    }
}

// kSpan: P.zspan is set and receives the node layers the lookups read.  kNarrow: tiles other than 8x4.
template <int LAYOUT, bool kPolish, bool kSpan, bool kNarrow>
__global__ void __launch_bounds__(kThreads) relax_scan_kernel(const RelaxLaunch P) {
    int i, j, tx, ty;
    scan_pixel<kNarrow>(P, i, j, tx, ty);
    if (LAYOUT == 0 && tx >= 0) prefetch_tile_slab<kNarrow>(P, tx, ty, threadIdx.x);
    const int2 span = relax_pixel<LAYOUT, false, false, false, kPolish, kSpan>(P, P, i, j);
    if constexpr (kSpan) record_zspan(P, span);
}

// Tricubic energy grid (linear layout).
template <bool kPolish, bool kSpan, bool kNarrow>
__global__ void __launch_bounds__(kThreads) relax_scan_tricubic_kernel(const RelaxLaunch P) {
    int i, j, tx, ty;
    scan_pixel<kNarrow>(P, i, j, tx, ty);
    if (tx >= 0) prefetch_tile_slab<kNarrow>(P, tx, ty, threadIdx.x);
    const int2 span = relax_pixel<0, false, true, false, kPolish, kSpan>(P, P, i, j);
    if constexpr (kSpan) record_zspan(P, span);
}

// Pixels per warp.  A column is a serial chain, and its warp stops for every height change and cell
// reload of its other lanes, so a scan that leaves the GPU idle runs narrower warps: the narrowest tile
// (8x4, 4x4, 4x2, 2x2, 2x1, 1 pixels) that needs at most `per_sm` warps per SM, beyond which the issue
// slots the idle lanes waste cost more than the shorter chains save.  Which warp runs a pixel never
// changes its value.  Measured alone on 20 heights (us; 8x4 tiles -> the tile taken, and the next
// narrower one where that is the line): force grid 20^2 px 274 -> 126 (1 px), 40^2 252 -> 146 (4),
// 64^2 226 -> 162 (8), 96^2 207 -> 179 (16), 128^2 199 (32; 16: 189, but 131 against 110 per scan with
// four in flight); with Newton polish, whose chains are longer, 40^2 638 -> 213 (2), 128^2 596 -> 543
// (16); energy grid 64^2 292 -> 229 (8; 4: 246), 128^2 296 (32; 16: 310).
void tile_shape(RelaxLaunch& L, int sms) {
    int lanes = L.tile_lanes;
    if (lanes <= 0) {
        const long long per_sm = (L.polish > 0 && L.map.interp == 0) ? 8 : 4;
        const long long npix = (long long)L.snx * L.sny;
        for (lanes = 1; lanes < 32 && (npix + lanes - 1) / lanes > per_sm * sms;) lanes *= 2;
    }
    for (;; lanes *= 2) {
        L.tile_wsh = lanes >= 32 ? 3 : lanes >= 8 ? 2 : lanes >= 2 ? 1 : 0;
        L.tile_hsh = lanes >= 16 ? 2 : lanes >= 4 ? 1 : 0;
        // (a grid holds 65535 tiles along y)
        if (lanes >= 32 || (L.sny - 1) >> L.tile_hsh < 65535) return;
    }
}

template <bool kPolish, bool kSpan, bool kNarrow>
void launch_relax_scan_n(const RelaxLaunch& L, dim3 grid, cudaStream_t s) {
    if (L.map.interp == 1) relax_scan_tricubic_kernel<kPolish, kSpan, kNarrow><<<grid, kThreads, 0, s>>>(L);
    else if (L.layout == 0) relax_scan_kernel<0, kPolish, kSpan, kNarrow><<<grid, kThreads, 0, s>>>(L);
    else relax_scan_kernel<1, kPolish, kSpan, kNarrow><<<grid, kThreads, 0, s>>>(L);
}

template <bool kPolish, bool kSpan>
void launch_relax_scan_t(const RelaxLaunch& L, dim3 grid, cudaStream_t s) {
    if (L.tile_wsh == 3 && L.tile_hsh == 2) launch_relax_scan_n<kPolish, kSpan, false>(L, grid, s);
    else launch_relax_scan_n<kPolish, kSpan, true>(L, grid, s);
}

}  // namespace

cudaError_t launch_relax_scan(const RelaxLaunch& L0, cudaStream_t s) {
    RelaxLaunch L = L0;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    tile_shape(L, sms);
    dim3 grid((L.snx + (1 << L.tile_wsh) - 1) >> L.tile_wsh, (L.sny + (1 << L.tile_hsh) - 1) >> L.tile_hsh, 1);
    if (L.plan_list) grid = dim3(L.plan_hblocks + grid.x * grid.y, 1, 1);
    const bool span = L.zspan != nullptr;
    if (L.polish > 0) span ? launch_relax_scan_t<true, true>(L, grid, s) : launch_relax_scan_t<true, false>(L, grid, s);
    else span ? launch_relax_scan_t<false, true>(L, grid, s) : launch_relax_scan_t<false, false>(L, grid, s);
    return cudaGetLastError();
}

PP_CHECK_READER(check_flags_relax_scan)

}  // namespace pp
