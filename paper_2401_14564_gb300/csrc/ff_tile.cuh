// Force-field assembly of one 16x16x16-node tile of a grid by a CTA of 256 threads, shared by K1
// (ff_tile.cu) and the batch (batch.cu).
//
// The direct sum costs every node every atom, on FP32 pipes that are already busy.  But the field of an
// atom far from a block of nodes is smooth across it: over a tile of half extent h, the pair terms
// (poles at the atom, up to r^-14) of an atom at distance D >= 10 h from the tile's centre are
// polynomials of degree 7 per axis to FP32 rounding.  So the atoms are split per tile:
//   far   D >= max(10 h, 1.75 R_iPP) (and, see tile_far, no image switch and no coul_rc crossing inside
//         the tile): summed at the 8x8x8 Chebyshev points of the tile instead of its 4096 nodes, then
//         interpolated to the nodes along x, y and z (barycentric Lagrange interpolation on the target
//         side; published as the cluster-particle treecode, Boateng & Krasny 2013);
//   near  everything else: summed at the nodes as before.
// Interpolation error, measured in FP64 at D = 10 h over directions: relative to the largest force in the tile 1.5e-9
// (Coulomb), 1.5e-7 (the r^-7 term) and 3.9e-6 (r^-13); relative to the node's own 1.5e-9, 4.7e-7 and 3.5e-5.  The
// last counts with its weight against the r^-7 term, (R/r)^6 <= 0.035 at the centre and 0.11 at the nearest node, hence
// the bound on D / R: a whole Lennard-Jones pair is good to 4.7e-7 of the node's own force at any R up to it.  The
// direct sum's own rounding (rsqrt to 2 ulp, raised to the 8th) is 5e-7 per pair, about as much.  Coordinates are taken relative to the tile's centre (formed as a
// float pair, the atoms' kept as float pairs), which removes the rounding of absolute node coordinates that the
// direct kernel has; without the low parts the far sums would share an atom's rounding over a whole tile
// (flake 8.45e-7 against 8.0e-7 below).
//
// Measured (direct sums -> tiles, Simulator.make_ff): 60-atom flake on 256x256x200 nodes, forces only, 0.408
// -> 0.136 ms (the grid's 210 MB alone take 31 us); 40-atom molecule on 176x160x60 with the tip's quadrupole
// 76 -> 45 us; 97 atoms, energies only at 0.15 A, 160 -> 60 us; the 2516-atom slab on 512x512x250 109 ->
// 22.5 ms.  FP32 pipes set the pace as before.  Error against FP64, mean over layers of the relative
// 2-norm: 8.1e-7 -> 8.0e-7 (flake), 3.0e-7 -> 2.9e-7 (molecule), 7.3e-7 -> 4.2e-7 (800-atom periodic sheet).
//
// Why 16 nodes and 8 points: 8 points keep the far sum at 1/8 of the direct one (64 columns of 8 points
// fill two warps exactly, four atom groups a CTA); 24 nodes and 10 points, or 16 and 7, need D of 8.4 and
// 9.4 A at 0.1 A instead of 7.5, and lose in near atoms what they gain.  A tile with fewer than
// kFarMin far atoms sums them at the nodes too (the interpolation's fixed cost is about 7 atoms' direct cost).
#pragma once

#include "ff_core.cuh"

namespace pp {

constexpr int kTileN = 16;        // nodes per tile side
constexpr int kTileP = 8;         // interpolation points per side
constexpr int kTileThreads = 256;
constexpr int kTileChunk = 256;   // atoms classified per pass: one per thread
constexpr int kFarMin = 8;

namespace tile_detail {
// Chebyshev points cos((2m + 1) pi / 16) on [-1, 1], ascending.
constexpr double kCheb[kTileP] = {-0.98078528040323044913, -0.83146961230254523708, -0.55557023301960222474,
                                  -0.19509032201612826785, 0.19509032201612826785,  0.55557023301960222474,
                                  0.83146961230254523708,  0.98078528040323044913};
// The interpolation runs on differences from point kRef of each axis, f_ref + sum w_m (f_m - f_ref): the
// weights then sum to one exactly and the rounding of the products scales with the field's variation
// over the tile, not with the field.
constexpr int kRef = 3;
struct Weights {
    float w[kTileN][kTileP];            // w[k][m]: Lagrange basis m at node k; 1 for m = kRef
    float z[kTileN / 2][kTileP][2];     // the same for node pairs: (w[2t][m], w[2t + 1][m])
    float at[kTileP];                   // the points, in nodes from the centre
    float l[kTileN][kTileP];            // w without the differences: l[k][m] Lagrange basis m at node k
};
constexpr Weights make_weights() {
    Weights r{};
    for (int m = 0; m < kTileP; ++m) r.at[m] = (float)(kCheb[m] * (0.5 * (kTileN - 1)));
    for (int k = 0; k < kTileN; ++k) {
        const double u = (k - 0.5 * (kTileN - 1)) / (0.5 * (kTileN - 1));
        for (int m = 0; m < kTileP; ++m) {
            double l = 1.0;
            for (int j = 0; j < kTileP; ++j)
                if (j != m) l *= (u - kCheb[j]) / (kCheb[m] - kCheb[j]);
            r.l[k][m] = (float)l;
            if (m == kRef) l = 1.0;
            r.w[k][m] = (float)l;
            r.z[k / 2][m][k & 1] = (float)l;
        }
    }
    return r;
}
}  // namespace tile_detail

namespace {
__constant__ tile_detail::Weights c_tile = tile_detail::make_weights();      // for indices a warp shares
__device__ const tile_detail::Weights g_tile = tile_detail::make_weights();  // for indices by thread
}  // namespace

// Grid and atoms of one assembly, as the tile needs them.
struct TileJob {
    const float *x, *y, *z, *R, *eps, *q;
    int n;
    float x0, y0, z0, dx, dy, dz;
    int nx, ny;
};

struct TileShared {
    // phase A: far records (first half); then the four groups' partial sums (all of it); then phase B's
    // x-interpolated values (second half) beside phase C's near records (first half)
    float4 buf[4 * kTileP * kTileP * kTileP];
    float4 sum[kTileP * kTileP * kTileP];
    int count[2][kTileThreads / 32];
};
static_assert(sizeof(float4) * 2 * kTileP * kTileP * kTileP >= 4 * sizeof(float4) * kTileChunk, "records fit");
static_assert(kTileN * kTileP * kTileP <= 2 * kTileP * kTileP * kTileP, "x-interpolated values fit");

// Centre of the tile's nodes along one axis, origin + (first + 7.5) d, as a float pair.
__device__ __forceinline__ float2 tile_centre(float origin, int first, float d) {
    const float m = __fadd_rn((float)first, 0.5f * (kTileN - 1));  // exact below 2^22 nodes
    const float p = __fmul_rn(m, d), pl = __fmaf_rn(m, d, -p);
    float s, e;
    two_sum(origin, p, s, e);
    return make_float2(s, __fadd_rn(e, pl));
}

// An atom's coordinate relative to the centre as a float pair (an infinite difference has no low part: its error term
// is not a number).
__device__ __forceinline__ void tile_rel(float a, float2 ctr, float& hi, float& lo) {
    float e;
    two_sum(a, -ctr.x, hi, e);
    lo = fabsf(hi) < 3.4e38f ? __fsub_rn(e, ctr.y) : 0.f;
}

// The same rounded once.
__device__ __forceinline__ float centred(float a, float2 ctr) {
    float hi, lo;
    tile_rel(a, ctr, hi, lo);
    return __fadd_rn(hi, lo);
}

__device__ __forceinline__ float wrap_image(float d, float L, float invL) { return __fmaf_rn(-L, rintf(__fmul_rn(d, invL)), d); }

// Whether the atom at (rx, ry, rz) from the tile's centre is summed at the interpolation points; on true,
// *charged tells whether its point-charge terms act inside the tile (with coul_rc: the whole tile lies
// within it) or nowhere (the whole tile beyond).  Explicit roundings: every kernel decides alike.
template <bool kMinImage, bool kCutoff>
__device__ __forceinline__ bool tile_far(const FFConst& c, float rx, float ry, float rz, float hx, float hy, float hz,
                                         float hmax, float R, float eps, float q, bool* charged) {
    const float ax = fabsf(rx), ay = fabsf(ry), az = fabsf(rz);
    const float d2 = __fmaf_rn(rx, rx, __fmaf_rn(ry, ry, __fmul_rn(rz, rz)));
    const float Rij = __fadd_rn(R, c.R_pp);
    // (the pair terms and the core floor take R_iPP squared: a sum below zero reaches as far)
    const float reach = fmaxf(__fmul_rn(10.f, hmax), __fmul_rn(1.75f, fabsf(Rij)));
    *charged = true;
    // (a coordinate, radius, depth or charge that is not finite: near, as the direct sum has it)
    if (!(d2 >= __fmul_rn(reach, reach)) || !(d2 < 3.0e38f)) return false;
    if (!(fabsf(Rij) < 3.0e38f) || !(fabsf(q) < 3.0e38f) || !(fabsf(eps) < 3.0e38f)) return false;
    if (kMinImage) {
        // some node of the tile sees another image of the atom
        if (!(__fadd_rn(ax, hx) < __fmul_rn(0.4999f, c.Lx)) || !(__fadd_rn(ay, hy) < __fmul_rn(0.4999f, c.Ly))) return false;
    }
    if (kCutoff && q != 0.f) {
        const float nx = fmaxf(__fsub_rn(ax, hx), 0.f), ny = fmaxf(__fsub_rn(ay, hy), 0.f), nz = fmaxf(__fsub_rn(az, hz), 0.f);
        const float fx = __fadd_rn(ax, hx), fy = __fadd_rn(ay, hy), fz = __fadd_rn(az, hz);
        const float dmin2 = __fmaf_rn(nx, nx, __fmaf_rn(ny, ny, __fmul_rn(nz, nz)));
        const float dmax2 = __fmaf_rn(fx, fx, __fmaf_rn(fy, fy, __fmul_rn(fz, fz)));
        if (dmin2 > __fmul_rn(1.0001f, c.rc2)) *charged = false;
        else if (!(dmax2 < __fmul_rn(0.9999f, c.rc2))) return false;
    }
    return true;
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 sub4(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }

// Slot of this thread's atom in an ordered compaction over the CTA (two barriers); *total: atoms kept.
__device__ __forceinline__ int tile_slot(bool keep, int* count, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned mask = __ballot_sync(0xffffffffu, keep);
    __syncthreads();  // the records and counts of the pass before have been read
    if (lane == 0) count[warp] = __popc(mask);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kTileThreads / 32; ++w) {
        const int c = count[w];
        before += w < warp ? c : 0;
        all += c;
    }
    *total = all;
    return before + __popc(mask & ((1u << lane) - 1u));
}

// Assembles the nodes of the tile at node (i0, j0, k0) (multiples of 16) and hands each thread's columns
// to `store(i, j, k, fx, fy, fz, en)`: node pairs (k, k + 1) of column (i, j) as packed pairs, for the halves of the
// tile that `want(first, count)` asks layers of (k0 + first .. k0 + first + count - 1), or with kThin, where one or two
// quarters of four layers are asked for, for those (the kernel that can do both is 3 % slower on whole grids).  Every
// thread of the CTA calls.
// A thread owns a column of 16 nodes, so that an atom's lateral terms and the interpolation along y
// are formed once for all of them (the two halves in turn, at fewer registers and three CTAs an SM: 0.142
// against 0.135 ms on the 60-atom flake, 24.2 against 22.2 ms on the slab).
template <bool kMinImage, bool kCutoff, bool kQuad, bool kEnergy, bool kForcesOnly, bool kThin, class Want, class Store>
__device__ __forceinline__ void ff_tile(const TileJob& J, const FFConst& c, int i0, int j0, int k0, TileShared& S,
                                        Want&& want, Store&& store) {
    constexpr int P3 = kTileP * kTileP * kTileP;
    const int tid = threadIdx.x;
    const float2 cx = tile_centre(J.x0, i0, J.dx), cy = tile_centre(J.y0, j0, J.dy), cz = tile_centre(J.z0, k0, J.dz);
    const float half = 0.5f * (kTileN - 1);
    const float hx = __fmul_rn(half, J.dx), hy = __fmul_rn(half, J.dy), hz = __fmul_rn(half, J.dz);
    const float hmax = fmaxf(hx, fmaxf(hy, hz));
    float4* const r0 = S.buf;
    float4* const r1 = r0 + kTileChunk;
    float4* const r2 = r1 + kTileChunk;
    float4* const r3 = r2 + kTileChunk;
    const bool one_chunk = J.n <= kTileChunk;

    struct Atom {
        float x, y, z, R, eps, q;
        float xl, yl, zl;
        bool live, far, charged;
    };
    auto load = [&](int a) {
        Atom t;
        t.live = a < J.n;
        t.far = false;
        t.charged = true;
        t.x = t.y = t.z = t.R = t.eps = t.q = t.xl = t.yl = t.zl = 0.f;
        if (t.live) {
            tile_rel(__ldg(J.x + a), cx, t.x, t.xl);
            tile_rel(__ldg(J.y + a), cy, t.y, t.yl);
            tile_rel(__ldg(J.z + a), cz, t.z, t.zl);
            if (kMinImage) {
                t.x = wrap_image(t.x, c.Lx, c.invLx);
                t.y = wrap_image(t.y, c.Ly, c.invLy);
            }
            t.R = __ldg(J.R + a);
            t.eps = __ldg(J.eps + a);
            t.q = __ldg(J.q + a);
            t.far = tile_far<kMinImage, kCutoff>(c, t.x, t.y, t.z, hx, hy, hz, hmax, t.R, t.eps, t.q, &t.charged);
        }
        return t;
    };
    auto stage = [&](const Atom& t, int slot, bool charged, bool far) {
        ff_stage_atom(c, t.x, t.y, t.z, t.R, t.eps, charged ? t.q : 0.f, r0[slot], r1[slot], r2[slot], r3[slot]);
        r1[slot].y = t.xl;
        r3[slot].y = t.yl;
        r3[slot].w = far ? 2.f * t.z * t.zl : -t.zl;
    };

    // ---- A: far atoms at the interpolation points
    const int group = tid >> 6, col = tid & 63;  // column (col & 7, col >> 3), atoms group, group + 4, ...
    float2 ax[4], ay[4], az[4], ae[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) ax[t] = ay[t] = az[t] = ae[t] = make_float2(0.f, 0.f);
    bool use_far = false;
    {
        float2 gz[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)
            gz[t] = make_float2(__fmul_rn(c_tile.at[2 * t], J.dz), __fmul_rn(c_tile.at[2 * t + 1], J.dz));
        const float gx = __fmul_rn(g_tile.at[col & 7], J.dx), gy = __fmul_rn(g_tile.at[col >> 3], J.dy);
        for (int base = 0; base < J.n; base += kTileChunk) {
            const Atom t = load(base + tid);
            // with a cutoff the charged atoms come first, then those without point-charge terms here
            const bool plain = kCutoff && !(t.charged && t.q != 0.f);
            int total, nq = 0;
            int slot = tile_slot(t.far && !plain, S.count[0], &nq);
            total = nq;
            if (kCutoff) {
                int np;
                const int sp = tile_slot(t.far && plain, S.count[0], &np);
                if (plain) slot = nq + sp;
                total = nq + np;
            }
            if (one_chunk ? total < kFarMin : total == 0) continue;
            use_far = true;
            if (t.far) stage(t, slot, t.charged, true);
            __syncthreads();
            // this group's atoms lie side by side: a quarter of each kind
            auto sum = [&](auto smooth, int from, int cnt) {
                const int first = from + ((cnt * group) >> 2), last = from + ((cnt * (group + 1)) >> 2);
                ff_accumulate_impl<4, false, kCutoff, kQuad, false, false, decltype(smooth)::value, true>(
                    r0 + first, r1 + first, r2 + first, r3 + first, last - first, c, gx, gy, gz, ax, ay, az, ae, ax, ay, az, ae);
            };
            sum(std::integral_constant<Smooth, Smooth::kInside>{}, 0, nq);
            if (kCutoff) sum(std::integral_constant<Smooth, Smooth::kBeyond>{}, nq, total - nq);
        }
    }

    // ---- B: the four groups' sums added, then interpolated along x
    float4* const X = S.buf + 2 * P3;  // [z point][y point][node along x]
    if (use_far) {
        // differences from the reference point along z, in registers: every thread has its column's points
        auto along_z = [](float2 (&a)[4]) {
            const float ref = (tile_detail::kRef & 1) ? a[tile_detail::kRef / 2].y : a[tile_detail::kRef / 2].x;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (2 * t != tile_detail::kRef) a[t].x -= ref;
                if (2 * t + 1 != tile_detail::kRef) a[t].y -= ref;
            }
        };
        along_z(ax); along_z(ay); along_z(az); along_z(ae);
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            // (sums that are not asked for are not formed: the compiler drops them with their stores)
            const float2 vx = kEnergy ? make_float2(0.f, 0.f) : ax[t], vy = kEnergy ? make_float2(0.f, 0.f) : ay[t];
            const float2 vz = kEnergy ? make_float2(0.f, 0.f) : az[t], ve = kForcesOnly ? make_float2(0.f, 0.f) : ae[t];
            S.buf[group * P3 + (2 * t) * 64 + col] = make_float4(vx.x, vy.x, vz.x, ve.x);
            S.buf[group * P3 + (2 * t + 1) * 64 + col] = make_float4(vx.y, vy.y, vz.y, ve.y);
        }
        __syncthreads();
        for (int e = tid; e < P3; e += kTileThreads) {
            float4 a = S.buf[e];
#pragma unroll
            for (int g = 1; g < 4; ++g) a = add4(a, S.buf[g * P3 + e]);
            S.sum[e] = a;
        }
        __syncthreads();
        // along y and x: point (m, n) of a z plane becomes (f_mn - f_mr) - (f_rn - f_rr), f_mr - f_rr, ...
        float4 d[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = tid + u * kTileThreads, px = e & 7, py = (e >> 3) & 7, plane = e & ~63;
            const float4 rx = S.sum[(e & ~7) + tile_detail::kRef], ry = S.sum[plane + tile_detail::kRef * 8 + px];
            const float4 rr = S.sum[plane + tile_detail::kRef * 9];
            float4 v = S.sum[e], w = ry;
            if (px != tile_detail::kRef) {
                v = sub4(v, rx);
                w = sub4(ry, rr);
            }
            d[u] = py != tile_detail::kRef ? sub4(v, w) : v;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) S.sum[tid + u * kTileThreads] = d[u];
        __syncthreads();
        const int i = tid & (kTileN - 1);
        float w[kTileP];
#pragma unroll
        for (int m = 0; m < kTileP; ++m) w[m] = g_tile.w[i][m];
        for (int row = tid >> 4; row < kTileP * kTileP; row += kTileThreads / kTileN) {
            float2 a = make_float2(0.f, 0.f), b = a;
#pragma unroll
            for (int m = 0; m < kTileP; ++m) {
                const float4 v = S.sum[row * kTileP + m];
                const float2 W = make_float2(w[m], w[m]);
                a = f2fma(W, make_float2(v.x, v.y), a);
                b = f2fma(W, make_float2(v.z, v.w), b);
            }
            X[row * kTileN + i] = make_float4(a.x, a.y, b.x, b.y);
        }
    }

    // ---- C: per column, the far field along y and z, then the near atoms at the nodes
    const int lane = tid & 31, warp = tid >> 5;
    const int i = (warp & 1) * 8 + (lane & 7), j = (warp >> 1) * 4 + (lane >> 3);
    const float gx = __fmul_rn((float)i - half, J.dx), gy = __fmul_rn((float)j - half, J.dy);
    float wy[kTileP];
    if (use_far) {
#pragma unroll
        for (int m = 0; m < kTileP; ++m) wy[m] = g_tile.w[j][m];
    }
    // ZP node pairs from layer k0 + first
    auto column = [&](auto zp, int first) {
        constexpr int ZP = decltype(zp)::value;
        float2 fx[ZP], fy[ZP], fz[ZP], en[ZP], gz[ZP];
#pragma unroll
        for (int t = 0; t < ZP; ++t) {
            fx[t] = fy[t] = fz[t] = en[t] = make_float2(0.f, 0.f);
            const float kk = (float)(first + 2 * t) - half;
            gz[t] = make_float2(__fmul_rn(kk, J.dz), __fmul_rn(kk + 1.f, J.dz));
        }
        if (use_far) {
            __syncthreads();  // X complete
#pragma unroll 2
            for (int m = 0; m < kTileP; ++m) {
                float2 a = make_float2(0.f, 0.f), b = a;
#pragma unroll
                for (int n = 0; n < kTileP; ++n) {
                    const float4 v = X[(m * kTileP + n) * kTileN + i];
                    const float2 W = make_float2(wy[n], wy[n]);
                    if (!kEnergy) a = f2fma(W, make_float2(v.x, v.y), a);
                    b = f2fma(W, make_float2(v.z, v.w), b);
                }
#pragma unroll
                for (int t = 0; t < ZP; ++t) {
                    const float2 W = make_float2(c_tile.z[(first >> 1) + t][m][0], c_tile.z[(first >> 1) + t][m][1]);
                    if (!kEnergy) {
                        fx[t] = f2fma(W, make_float2(a.x, a.x), fx[t]);
                        fy[t] = f2fma(W, make_float2(a.y, a.y), fy[t]);
                        fz[t] = f2fma(W, make_float2(b.x, b.x), fz[t]);
                    }
                    if (!kForcesOnly) en[t] = f2fma(W, make_float2(b.y, b.y), en[t]);
                }
            }
        }
        for (int base = 0; base < J.n; base += kTileChunk) {
            const Atom t = load(base + tid);
            const bool near = t.live && !(use_far && t.far);
            int total;
            const int slot = tile_slot(near, S.count[1], &total);
            if (near) stage(t, slot, true, false);
            __syncthreads();
            ff_accumulate_impl<ZP, kMinImage, kCutoff, kQuad, false, true, Smooth::kNo, true>(r0, r1, r2, r3, total, c, gx, gy, gz, fx, fy,
                                                                          fz, en, fx, fy, fz, en);
        }
#pragma unroll
        for (int t = 0; t < ZP; ++t) store(i0 + i, j0 + j, k0 + first + 2 * t, fx[t], fy[t], fz[t], en[t]);
    };
    const std::integral_constant<int, 8> whole;
    const std::integral_constant<int, 4> half_tile;
    const std::integral_constant<int, 2> quarter;
    if constexpr (kThin) {
        int q0 = 0, q1 = 4;
        while (q0 < 3 && !want(4 * q0, 4)) ++q0;
        while (q1 > q0 + 1 && !want(4 * q1 - 4, 4)) --q1;
        if (q1 - q0 > 2) column(whole, 0);
        else if (q1 - q0 == 2) column(half_tile, 4 * q0);
        else column(quarter, 4 * q0);
    } else {
        if (want(0, 8) && want(8, 8)) column(whole, 0);
        else if (want(0, 8)) column(half_tile, 0);
        else if (want(8, 8)) column(half_tile, 8);
    }
    __syncthreads();  // the shared buffers may be reused
}

// ---- which way a grid is assembled
// One rounding per operation on the device and on the host, whose compiler may fuse: K1's launcher and the batch kernel
// decide alike.
__host__ __device__ inline float rule_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    const volatile float r = a * b;
    return r;
#endif
}
__host__ __device__ inline float rule_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    const volatile float r = a + b;
    return r;
#endif
}
__host__ __device__ inline float rule_sqrt(float a) {
#ifdef __CUDA_ARCH__
    return __fsqrt_rn(a);
#else
    return sqrtf(a);
#endif
}

// Estimate of the share of (node, atom) pairs at `reach` and more, for atoms spread over the cell Lx x Ly in a plane
// 3 A below the grid (a molecule's depth and the grid's clearance): at each of eight heights those outside a disc of
// radius sqrt(reach^2 - h^2), of which a narrow cell holds a strip at most.
__host__ __device__ inline float ff_far_share(float Lx, float Ly, float Lz, float reach) {
    const float area = rule_mul(Lx, Ly), r2 = rule_mul(reach, reach), side = Lx < Ly ? Lx : Ly;
    float sum = 0.f;
    for (int i = 0; i < 8; ++i) {
        const float h = rule_add(3.f, rule_mul((i + 0.5f) * 0.125f, Lz)), d2 = rule_add(r2, -rule_mul(h, h));
        if (!(d2 > 0.f)) {
            sum = rule_add(sum, 1.f);
            continue;
        }
        const float disc = rule_mul(3.14159265f, d2), strip = rule_mul(2.f * rule_sqrt(d2), side);
        const float in = disc < strip ? disc : strip;
        if (in < area) sum = rule_add(sum, rule_add(1.f, -(in / area)));
    }
    return 0.125f * sum;
}

// kDirect: direct sums.  Few atoms: they cost less than a tile's classification and, where a tile has them,
// interpolation (160x160x60 nodes at 0.1 A, whole call: 16 atoms 29 us directly, 23 by tiles; 24 atoms 38 and 29;
// 10 atoms 23 directly, where the call's own 20 us already show).  Coarse grids: beyond 0.35 A no atom nearer
// than 26 A is far, and coordinates relative to the centre of a wide tile round worse than absolute ones.  And where a
// tile would find little far, so that its classification, the float pairs of its coordinates and its coarser blocks
// show: energies alone (whose direct sums are half as long) where the share of far pairs is below 0.4, and fewer than 36
// atoms where it is below 0.3.  Measured on either side of the line (K1 alone, us: direct sums / tiles):
//   energies: 198 atoms on 61x111x53 nodes (0.2 A, share 0.06) 44 / 55; 43 on 149x120x56 (0.2 A, 0.38) 23 / 27; 49 on
//   86x154x46 (0.1 A, 0.43) 20 / 18; 493 on 129x124x42 (0.1 A, 0.43) 193 / 94; 84 on 61x219x60 (0.2 A, 0.51) 52 / 45;
//   32 atoms on 105x66x40 (0.1 A, 0.10) 20 / 23; 28 on 105x65x69 (0.2 A, 0.24) 16 / 20; 33 on 76x229x97 (0.2 A, 0.71) 47 / 35;
//   with more atoms 46 on 118x85x54 (0.1 A) 29 / 25.  (Between 0.3 and 0.6 few atoms' direct sums are up to 15 % faster alone,
//   but the batch, which must write the same bits by 16-node tiles, loses 2 to 5 %: 4 molecules at 84 px 756 -> 798.)
// kCentred: direct sums with coordinates relative to the tile's centre, on periodic cells where that share is below 0.3
// (energies 0.4; absolute coordinates / tiles / centred): 148 atoms on 71x215x73 (0.28 A, 0.00) 182 / 253 / 176; 184 on 106x340x85 (0.21 A,
// 0.07) 430 / 513 / 415; 420 on 354x134x147 (0.29 A, 0.17) 2414 / 2578 / 2427; 380 on 124x386x153 (0.26 A, 0.31)
// 1740 / 1632 / 1754; 172 on 146x193x53 (0.15 A, 0.37) 213 / 222 / 199; 228 on 281x111x196 (0.23 A, 0.44) 1090 / 897 / 1113.
// Their coordinates round once, which keeps most of what the tiles gain in accuracy there (relative 2-norm of the error
// against FP64, 124-atom sheet on 71x124x95: 7.7e-7 / 6.2e-7 / 6.8e-7; low parts in every pair, as the tiles have them, cost
// 4 to 6 % of the time).  Molecules keep absolute coordinates: an atom's rounding is common to a tile's nodes, and about
// a wide tile it exceeds theirs (99 atoms' energies at 0.25 A 7.9e-7 / 8.0e-7 / 9.3e-7).
enum class FFPath { kDirect, kCentred, kTiles };
__host__ __device__ inline bool ff_tiles_possible(int n, float dx, float dy, float dz) {
    return n >= 16 && dx <= 0.35f && dy <= 0.35f && dz <= 0.35f;
}
__host__ __device__ inline FFPath ff_path(int n, int nx, int ny, int nz, float dx, float dy, float dz, bool min_image,
                                          bool energy) {
    if (!ff_tiles_possible(n, dx, dy, dz)) return FFPath::kDirect;
    if (!min_image && !energy && n >= 36) return FFPath::kTiles;
    const float dmax = dx > dy ? (dx > dz ? dx : dz) : (dy > dz ? dy : dz);
    const float reach = rule_mul(5.f * (kTileN - 1), dmax);  // 10 half extents
    const float share = ff_far_share(rule_mul((float)nx, dx), rule_mul((float)ny, dy), rule_mul((float)nz, dz), reach);
    if (share >= (energy ? 0.4f : 0.3f)) return FFPath::kTiles;
    return min_image ? FFPath::kCentred : FFPath::kDirect;
}

}  // namespace pp
