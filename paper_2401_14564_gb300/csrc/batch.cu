// K6: many molecules in one call (force field -> relaxed scan -> df per molecule, exactly the
// single-molecule path of K1 + K2): a planning kernel and two persistent ones.
//
// Work items:  FF tile    = 16x16x16 nodes of one molecule's grid, taken by a CTA of 256 threads;
//              relax tile = rw x (32/rw) pixels x all heights of one molecule, taken by a warp
// (rw in {4, 8, 16}: the shape changes the schedule, never a value).  Workers take the next item index from
// a device counter; the item list is FF(0), ..., FF(n-1), R(0), ..., R(n-1) (prefix sums built by the
// planning kernel).  Many molecules' tiles are in flight at once, which fills the GPU even though one
// 128x128 scan is only 512 warps.  The force fields are assembled by one kernel and scanned by the next:
// with the far atoms interpolated (ff_tile.cuh) assembly is a CTA's work, and what it takes is no longer
// enough to hide scans behind; a grid written to HBM and read back in its scan's layers costs 1 % of a
// batch's time.  A relax tile checks its molecule's count of finished force-field tiles (one that is short sets a status
// bit and the warp stops).
#include <cstring>

#include "ff_tile.cuh"
#include "relax_core.cuh"

namespace pp {
namespace {

constexpr int kThreads = 128;  // relax kernel: 4 independent warps per CTA
constexpr int kMinCtas = 5;    // resident CTAs per SM the register budget is sized for

struct BatchLaunch {
    const pp_mol_desc* descs;
    int nmol;
    const float *ax, *ay, *az, *aR, *aeps, *aq;
    int n_atoms_total;
    float4* ff;
    long long ff_cap;
    float *pos, *fz, *df;
    int* iters;
    long long out_cap, df_cap;
    // probe (shared)
    float R_pp, eps_pp, kQ, core_frac, coul_rc, kQzz;
    int min_image, periodic_xy;
    // tip, FIRE and df stencil, under the names relax_pixel expects
    float kx, ky, kR, R0, d0x, d0y, d0z, R0sq, c0;
    int max_iter, n_min;
    float ftol2, dt0, dt_max, f_inc, f_dec, alpha0, f_alpha, inv_mass;
    float sdz;
    int df_m;
    const float* coef;  // in ws, written by the planning kernel
    // scratch
    unsigned long long *counter_ff, *counter_relax;
    int* status;
    long long* seg_start;  // [2 nmol + 1]: first item of FF(m) at m, of R(m) at nmol + m, their end
    int* done_ff;          // [nmol]
    float* coef_ws;
    int wait_extra;
    int forces_only;  // E slots written as 0, energy sums skipped
    int rw_sh;        // log2 of the relax tile width (4, 8 or 16 lanes along x)
    float coef_init[2 * kMaxDfHalfWidth + 1];
};

// Per-molecule geometry for relax_pixel (linear layout).
struct MolRelax {
    const float4* ff;
    GridMap map;
    float inv_dx, inv_dy, inv_dz, gx0s, gy0s, gz0s;
    float fz0, fz0_lo, st, st_lo;
    int periodic_xy;
    int snx, sny, snz;
    float sx0, sy0, spx, spy, z_top;
    float *pos, *fz, *df;
    int* iters;
};

__device__ __forceinline__ long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

__device__ __forceinline__ long long ff_tiles(const pp_mol_desc& D) {
    return cdiv(D.nx, kTileN) * cdiv(D.ny, kTileN) * cdiv(D.nz, kTileN);
}
__device__ __forceinline__ long long relax_tiles(const BatchLaunch& B, const pp_mol_desc& D) {
    return cdiv(D.snx, 1 << B.rw_sh) * cdiv(D.sny, 32 >> B.rw_sh);
}

__device__ __forceinline__ bool finite_pos(float v) { return isfinite(v) && v > 0.f; }

// Every index a molecule's tiles will touch lies inside the caller's buffers.
__device__ bool mol_valid(const BatchLaunch& B, const pp_mol_desc& D) {
    if (D.nx < 2 || D.ny < 2 || D.nz < 2 || !finite_pos(D.dx) || !finite_pos(D.dy) || !finite_pos(D.dz)) return false;
    if (D.nx > (1 << 22) || D.ny > (1 << 22) || D.nz > (1 << 22)) return false;  // the cell lookup's fast floor
    if (!isfinite(D.x0) || !isfinite(D.y0) || !isfinite(D.z0)) return false;
    const long long nodes = (long long)D.nx * D.ny * D.nz;
    if (nodes >= (1LL << 31) || D.ff_offset < 0 || D.ff_offset + nodes > B.ff_cap) return false;
    if (D.n_atoms < 0 || D.atom_offset < 0 || (long long)D.atom_offset + D.n_atoms > B.n_atoms_total) return false;
    if (D.snx < 1 || D.sny < 1 || D.snz < 2 * B.df_m + 1) return false;
    if (!isfinite(D.sx0) || !isfinite(D.sy0) || !isfinite(D.spx) || !isfinite(D.spy) || !isfinite(D.z_top)) return false;
    const long long pts = (long long)D.snx * D.sny * D.snz;
    if (3 * pts >= (1LL << 31) || D.out_offset < 0 || D.out_offset + pts > B.out_cap) return false;
    const long long dfn = (long long)D.snx * D.sny * (D.snz - 2 * B.df_m);
    if (D.df_offset < 0 || D.df_offset + dfn > B.df_cap) return false;
    return true;
}

__global__ void __launch_bounds__(1024) batch_plan_kernel(const BatchLaunch B) {
    __shared__ long long wsum[32];
    __shared__ long long carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        *B.counter_ff = 0ULL;
        *B.counter_relax = 0ULL;
        *B.status = 0;
        carry = 0;
    }
    for (int c = tid; c < 2 * B.df_m + 1; c += blockDim.x) B.coef_ws[c] = B.coef_init[c];
    for (int m = tid; m < B.nmol; m += blockDim.x) B.done_ff[m] = 0;
    __syncthreads();
    const int nseg = 2 * B.nmol;
    for (int base = 0; base < nseg; base += blockDim.x) {
        const int s = base + tid;
        long long len = 0;
        if (s < nseg) {
            const bool ff = s < B.nmol;
            const pp_mol_desc D = B.descs[ff ? s : s - B.nmol];
            if (mol_valid(B, D)) len = ff ? ff_tiles(D) : relax_tiles(B, D);
            else if (ff) atomicOr(B.status, PP_BATCH_BAD_DESC);
        }
        // inclusive block scan of len
        long long v = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[warp] = v;
        __syncthreads();
        if (warp == 0) {
            long long w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long u = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += u;
            }
            wsum[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        const long long before = carry + (warp > 0 ? wsum[warp - 1] : 0);
        if (s < nseg) B.seg_start[s] = before + v - len;
        __syncthreads();
        if (tid == 0) carry += wsum[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (tid == 0) B.seg_start[nseg] = carry;
}

// Segment holding item t among seg_start[first .. last): the last s with seg_start[s] <= t.
__device__ __forceinline__ int find_segment(const BatchLaunch& B, int first, int last, long long t) {
    int lo = first, hi = last - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.seg_start[mid] <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Node pairs of a column of molecule D, the force sums as ff_tile and the direct sums hand them over.
template <bool kForcesOnly>
struct MolStore {
    const BatchLaunch& B;
    const pp_mol_desc& D;
    __device__ __forceinline__ void operator()(int i, int j, int k, float2 fx, float2 fy, float2 fz, float2 en) const {
        if (i >= D.nx || j >= D.ny) return;
        const long long first = D.ff_offset + (long long)j * D.nx + i, plane = (long long)D.nx * D.ny;
        auto at = [&](int kk) { return checked(first + kk * plane, (long long)B.ff_cap, kChkGridWrite); };
        if (kForcesOnly) en = make_float2(0.f, 0.f);
        if (k < D.nz) B.ff[at(k)] = make_float4(fx.x, fy.x, fz.x, en.x);
        if (k + 1 < D.nz) B.ff[at(k + 1)] = make_float4(fx.y, fy.y, fz.y, en.y);
    }
};

// Direct sums (grids not assembled by tiles, see ff_path) of 8 layers from k0 of the 8x4 columns from
// (i0, j0), by one warp: the arithmetic of ff_assemble.cu, with `centre` relative to the centre of the tile at
// (it, jt, kt).  st: 4 x 32 records.
template <bool kMinImage, bool kCutoff, bool kQuad, class Store>
__device__ __forceinline__ void ff_direct(const BatchLaunch& B, const pp_mol_desc& D, const FFConst& cst, int i0, int j0,
                                          int k0, bool centre, int it, int jt, int kt, float4* st, Store&& store) {
    constexpr int ZP = 4;
    constexpr float half = 0.5f * (kTileN - 1);
    const int lane = threadIdx.x & 31, i = i0 + (lane & 7), j = j0 + (lane >> 3);
    if (!kMinImage) centre = false;
    const float gx = centre ? __fmul_rn((float)(i - it) - half, D.dx) : D.x0 + i * D.dx;
    const float gy = centre ? __fmul_rn((float)(j - jt) - half, D.dy) : D.y0 + j * D.dy;
    const float2 cx = tile_centre(D.x0, it, D.dx), cy = tile_centre(D.y0, jt, D.dy), cz = tile_centre(D.z0, kt, D.dz);
    float2 gz[ZP], fx[ZP], fy[ZP], fz[ZP], en[ZP];
#pragma unroll
    for (int t = 0; t < ZP; ++t) {
        const int k = k0 + 2 * t;
        gz[t] = centre ? make_float2(__fmul_rn((float)(k - kt) - half, D.dz), __fmul_rn((float)(k + 1 - kt) - half, D.dz))
                       : make_float2(D.z0 + k * D.dz, D.z0 + (k + 1) * D.dz);
        fx[t] = fy[t] = fz[t] = en[t] = make_float2(0.f, 0.f);
    }
    for (int base = 0; base < D.n_atoms; base += 32) {
        const int cnt = min(32, D.n_atoms - base);
        __syncwarp();
        if (lane < cnt) {
            const int g = D.atom_offset + base + lane;
            float x = B.ax[g], y = B.ay[g], z = B.az[g];
            if (kMinImage && centre) {
                x = wrap_image(centred(x, cx), cst.Lx, cst.invLx);
                y = wrap_image(centred(y, cy), cst.Ly, cst.invLy);
                z = centred(z, cz);
            }
            ff_stage_atom(cst, x, y, z, B.aR[g], B.aeps[g], B.aq[g], st[lane], st[32 + lane], st[64 + lane], st[96 + lane]);
        }
        __syncwarp();
        ff_accumulate<ZP, kMinImage, kCutoff, kQuad, true>(st, st + 32, st + 64, st + 96, cnt, cst, gx, gy, gz, fx, fy, fz,
                                                           en);
    }
#pragma unroll
    for (int t = 0; t < ZP; ++t) store(i, j, k0 + 2 * t, fx[t], fy[t], fz[t], en[t]);
}

template <bool kMinImage, bool kCutoff, bool kQuad, bool kForcesOnly>
__global__ void __launch_bounds__(kTileThreads, 2) batch_ff_kernel(const BatchLaunch B) {
    __shared__ TileShared S;
    __shared__ long long item;
    const long long total = B.seg_start[B.nmol];
    for (;;) {
        if (threadIdx.x == 0) item = (long long)atomicAdd(B.counter_ff, 1ULL);
        __syncthreads();
        const long long t = item;
        __syncthreads();
        if (t >= total) break;
        const int mol = find_segment(B, 0, B.nmol, t);
        const pp_mol_desc& D = B.descs[mol];
        const long long tile = t - B.seg_start[mol];
        const int tx_n = (D.nx + kTileN - 1) / kTileN, ty_n = (D.ny + kTileN - 1) / kTileN;
        const int tz = (int)(tile / ((long long)tx_n * ty_n));
        const int r = (int)(tile - (long long)tz * tx_n * ty_n);
        const int i0 = (r % tx_n) * kTileN, j0 = (r / tx_n) * kTileN, k0 = tz * kTileN;
        const FFConst cst = ff_const(B.R_pp, B.eps_pp, B.kQ, B.core_frac, D.nx * D.dx, D.ny * D.dy,
                                     kCutoff ? B.coul_rc : 0.f, kQuad ? B.kQzz : 0.f);
        const MolStore<kForcesOnly> store{B, D};
        const FFPath path = ff_path(D.n_atoms, D.nx, D.ny, D.nz, D.dx, D.dy, D.dz, kMinImage, false);
        if (path == FFPath::kTiles) {
            const int a = D.atom_offset;
            const TileJob J = {B.ax + a, B.ay + a, B.az + a, B.aR + a, B.aeps + a, B.aq + a, D.n_atoms,
                               D.x0, D.y0, D.z0, D.dx, D.dy, D.dz, D.nx, D.ny};
            const int nz = D.nz;
            ff_tile<kMinImage, kCutoff, kQuad, false, kForcesOnly, false>(J, cst, i0, j0, k0, S,
                                                                          [&](int f, int) { return k0 + f < nz; }, store);
        } else {
            const int warp = threadIdx.x >> 5;
            for (int h = 0; h < 2; ++h)
                if (k0 + 8 * h < D.nz)
                    ff_direct<kMinImage, kCutoff, kQuad>(B, D, cst, i0 + (warp & 1) * 8, j0 + (warp >> 1) * 4, k0 + 8 * h,
                                                         path == FFPath::kCentred, i0, j0, k0, S.buf + warp * 128, store);
        }
        if (threadIdx.x == 0) atomicAdd(B.done_ff + mol, 1);
    }
}

__global__ void __launch_bounds__(kThreads, kMinCtas) batch_relax_kernel(const BatchLaunch B) {
    const int lane = threadIdx.x & 31;
    const long long first = B.seg_start[B.nmol], total = B.seg_start[2 * B.nmol] - first;
    for (;;) {
        long long t = 0;
        if (lane == 0) t = (long long)atomicAdd(B.counter_relax, 1ULL);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= total) break;
        const int seg = find_segment(B, B.nmol, 2 * B.nmol, first + t), mol = seg - B.nmol;
        const long long tile = first + t - B.seg_start[seg];
        const pp_mol_desc D = B.descs[mol];
        // every force-field tile of this molecule is done, by stream order: a check, not a wait
        if (B.done_ff[mol] < (int)(B.seg_start[mol + 1] - B.seg_start[mol]) + B.wait_extra) {
            if (lane == 0) atomicOr(B.status, PP_BATCH_TIMEOUT);
            break;
        }
        MolRelax G;
        G.ff = B.ff + D.ff_offset;
        G.map.nx = D.nx; G.map.ny = D.ny; G.map.nz = D.nz;
        G.map.ax = {0, 1, 0, 0};
        G.map.ay = {0, D.nx, 0, 0};
        G.map.az = {0, D.nx * D.ny, 0, 0};
        G.map.stored_nodes = (int64_t)D.nx * D.ny * D.nz;
        G.map.interp = 0;
        G.inv_dx = 1.f / D.dx; G.inv_dy = 1.f / D.dy; G.inv_dz = 1.f / D.dz;
        G.gx0s = (float)(-(double)D.x0 / (double)D.dx);
        G.gy0s = (float)(-(double)D.y0 / (double)D.dy);
        G.gz0s = (float)(-(double)D.z0 / (double)D.dz);
        split_height_steps(D.z_top, B.d0z, B.sdz, D.z0, D.dz, &G.fz0, &G.fz0_lo, &G.st, &G.st_lo);
        G.periodic_xy = B.periodic_xy;
        G.snx = D.snx; G.sny = D.sny; G.snz = D.snz;
        G.sx0 = D.sx0; G.sy0 = D.sy0; G.spx = D.spx; G.spy = D.spy; G.z_top = D.z_top;
        G.fz = B.fz + D.out_offset;
        G.pos = B.pos ? B.pos + 3 * D.out_offset : nullptr;
        G.iters = B.iters ? B.iters + D.out_offset : nullptr;
        G.df = B.df + D.df_offset;
        const int rw = 1 << B.rw_sh;
        const int tiles_x = (D.snx + rw - 1) / rw;
        const int ty = (int)(tile / tiles_x), tx = (int)(tile - (long long)ty * tiles_x);
        relax_pixel<0, false, false, true>(G, B, tx * rw + (lane & (rw - 1)), ty * (32 >> B.rw_sh) + (lane >> B.rw_sh));
    }
}

}  // namespace

size_t batch_workspace_bytes(int nmol) {
    if (nmol < 1) return 0;
    const size_t b = 320 + 8 * (2 * (size_t)nmol + 1) + 4 * (size_t)nmol;
    return (b + 15) & ~size_t(15);
}

cudaError_t launch_batch(const BatchArgs& A, cudaStream_t s) {
    BatchLaunch B;
    memset(&B, 0, sizeof(B));
    B.descs = A.descs; B.nmol = A.nmol;
    B.ax = A.atoms.x; B.ay = A.atoms.y; B.az = A.atoms.z; B.aR = A.atoms.R; B.aeps = A.atoms.eps; B.aq = A.atoms.q;
    B.n_atoms_total = A.atoms.n;
    B.ff = reinterpret_cast<float4*>(A.ff);
    B.ff_cap = A.params.ff_capacity;
    B.pos = A.pos; B.fz = A.fz; B.df = A.df; B.iters = A.iters;
    B.out_cap = A.params.out_capacity; B.df_cap = A.params.df_capacity;
    const pp_batch_params& P = A.params;
    B.R_pp = P.probe.R_pp; B.eps_pp = P.probe.eps_pp;
    B.kQ = (float)(kCoulomb * (double)P.probe.Q);
    B.kQzz = (float)(0.5 * kCoulomb * (double)P.probe.Qzz);
    B.core_frac = P.probe.core_frac; B.coul_rc = P.probe.coul_rc;
    B.min_image = P.probe.min_image; B.periodic_xy = P.periodic_xy;
    B.kx = (float)(P.tip.kx * kNmToEvA2); B.ky = (float)(P.tip.ky * kNmToEvA2); B.kR = (float)(P.tip.kR * kNmToEvA2);
    B.R0 = P.tip.R0; B.d0x = P.tip.d0x; B.d0y = P.tip.d0y;
    B.d0z = (float)(-sqrt((double)P.tip.R0 * P.tip.R0 - (double)P.tip.d0x * P.tip.d0x -
                          (double)P.tip.d0y * P.tip.d0y));
    B.R0sq = (float)((double)P.tip.R0 * P.tip.R0);
    B.c0 = (float)((double)B.d0x * B.d0x + (double)B.d0y * B.d0y + (double)B.d0z * B.d0z -
                   (double)P.tip.R0 * P.tip.R0);
    B.max_iter = P.fire.max_iter; B.n_min = P.fire.n_min;
    B.ftol2 = P.fire.ftol * P.fire.ftol;
    B.dt0 = P.fire.dt0; B.dt_max = P.fire.dt_max; B.f_inc = P.fire.f_inc; B.f_dec = P.fire.f_dec;
    B.alpha0 = P.fire.alpha0; B.f_alpha = P.fire.f_alpha; B.inv_mass = 1.f / P.fire.mass;
    B.sdz = P.scan_dz;
    B.df_m = A.df_m;
    for (int c = 0; c < 2 * A.df_m + 1; ++c) B.coef_init[c] = A.coef[c];
    char* w = reinterpret_cast<char*>(A.ws);
    B.counter_ff = reinterpret_cast<unsigned long long*>(w);
    B.status = reinterpret_cast<int*>(w + 8);
    B.counter_relax = reinterpret_cast<unsigned long long*>(w + 16);
    B.coef_ws = reinterpret_cast<float*>(w + 64);
    B.coef = B.coef_ws;
    B.seg_start = reinterpret_cast<long long*>(w + 320);
    B.done_ff = reinterpret_cast<int*>(w + 320 + 8 * (2 * (size_t)A.nmol + 1));
    B.wait_extra = P.wait_extra;
    B.forces_only = P.ff_forces_only;
    const int rw = P.relax_tile_w > 0 ? P.relax_tile_w : 8;
    B.rw_sh = rw == 4 ? 2 : (rw == 8 ? 3 : 4);

    batch_plan_kernel<<<1, 1024, 0, s>>>(B);
    int dev = 0, sms = 152, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // (a caller's limit keeps the same SMs free of both kernels)
    const int ff_ctas = P.ctas > 0 && P.ctas < 2 * sms ? P.ctas : 2 * sms;
    with_flags(B.min_image != 0, B.coul_rc > 0.f, B.kQzz != 0.f, [&](auto mi, auto cut, auto quad) {
        constexpr bool MI = decltype(mi)::value, CUT = decltype(cut)::value, QUAD = decltype(quad)::value;
        if (B.forces_only) batch_ff_kernel<MI, CUT, QUAD, true><<<ff_ctas, kTileThreads, 0, s>>>(B);
        else batch_ff_kernel<MI, CUT, QUAD, false><<<ff_ctas, kTileThreads, 0, s>>>(B);
        return 0;
    });
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int ctas = P.ctas;
    if (ctas <= 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_relax_kernel, kThreads, 0);
        ctas = sms * (per_sm > 0 ? per_sm : 1);
    }
    batch_relax_kernel<<<ctas, kThreads, 0, s>>>(B);
    return cudaGetLastError();
}

PP_CHECK_READER(check_flags_batch)

}  // namespace pp
