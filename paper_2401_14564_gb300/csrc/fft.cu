// Cross-correlation force fields (Eqs. El_conv and Pauli_FDBM; Sec. 5.1.2:
// the convolution theorem turns the correlation into a product in Fourier
// space).  For a sample field f and a tip density g on the same periodic grid,
//   E[n] = scale * dV * sum_h g[h]^p f[n + h]^p,   F = -grad E,
// with the gradient taken spectrally (i k, Nyquist terms dropped so that the
// force stays real).  Steps, each one kernel, all in this file, with the bytes read + written per node:
//   x forward   z = f^p + i g^p (two real transforms in one complex one), formed while loading   8 + 8
//   y forward   in place                                                                         8 + 8
//   z middle    a CTA holds the lines (kx, ky) and (-kx, -ky): forward along z, then
//               F^ = (Z_k + Z*_-k)/2, G^ = (Z_k - Z*_-k)/(2i), P = G^* F^ scale dV / N, then P and
//               -i kz P inverse along z; E is real, so only kx = 0..nx/2 is kept from here on    8 + 8
//   y inverse   of P, -i ky P and -i kz P                                                        8 + 12
//   x inverse   rows of (E, Fx = -i kx E) and (Fy, Fz) as (re, im) of two complex transforms,
//               rebuilt from their halves while loading; ff[n] = (Fx, Fy, Fz, E), written or added  12 + 16
// 96 bytes per node; separate pack, spectral and output passes around nine full-spectrum ones moved 224.
// Measured: 512x512x128 nodes 1392 -> 870 us (3.7 TB/s of these bytes), with power 1.05 and accumulation 1582 -> 1085
// us, 128^3 139 -> 87 us, 32^3 52 -> 29 us (5 launches for 12).  Now bound by issue (61-78 % active in the
// first four kernels, 40 % in the last, which moves 28 of the 96 bytes).
// The 1D transforms are Stockham auto-sort FFTs with radix-8 stages (and one
// radix-2 or radix-4 stage) in registers, for power-of-two lengths up to 1024:
// a CTA transforms a tile of neighbouring lines (rows along x, columns along y
// and z, so every global access is a row of consecutive complex values); the
// first stage reads global memory, the last writes it, the ones between
// exchange through shared memory.
#include <cuda_runtime.h>

#include "fft_layout.cuh"
#include "pp_internal.cuh"

namespace pp {
namespace {

constexpr int kThreads = 256;
constexpr int kUnits = 2;          // stage units per thread per trip
constexpr int kLines = 16;         // lines per tile along x (at most)
constexpr int kStridedLines = 64;  // columns per tile along y and z (at most)

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a w, w = (cos, sin) of the positive angle, conjugated for SIGN = -1
template <int SIGN>
__device__ __forceinline__ float2 cmul(float2 w, float2 a) {
    const float s = SIGN > 0 ? w.y : -w.y;
    return make_float2(fmaf(w.x, a.x, -s * a.y), fmaf(w.x, a.y, s * a.x));
}
template <int SIGN>
__device__ __forceinline__ float2 mul_i(float2 a) { return SIGN > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x); }

// In-register DFT of R points (R = 2, 4, 8), natural order, w = exp(SIGN 2 pi i / R).
template <int R, int SIGN>
struct Dft;

template <int SIGN>
struct Dft<2, SIGN> {
    static __device__ __forceinline__ void run(float2 (&x)[2]) {
        const float2 a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};

template <int SIGN>
struct Dft<4, SIGN> {
    static __device__ __forceinline__ void run(float2 (&x)[4]) {
        const float2 t0 = cadd(x[0], x[2]), t1 = csub(x[0], x[2]);
        const float2 t2 = cadd(x[1], x[3]), t3 = mul_i<SIGN>(csub(x[1], x[3]));
        x[0] = cadd(t0, t2);
        x[2] = csub(t0, t2);
        x[1] = cadd(t1, t3);
        x[3] = csub(t1, t3);
    }
};

template <int SIGN>
struct Dft<8, SIGN> {
    static __device__ __forceinline__ void run(float2 (&x)[8]) {
        float2 e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
        Dft<4, SIGN>::run(e);
        Dft<4, SIGN>::run(o);
        const float h = 0.70710678118654752f, s = (float)SIGN;  // w8 = h (1 + sign i)
        const float2 o1 = make_float2(h * (o[1].x - s * o[1].y), h * (o[1].y + s * o[1].x));
        const float2 o2 = mul_i<SIGN>(o[2]);
        const float2 o3 = make_float2(h * (-o[3].x - s * o[3].y), h * (-o[3].y + s * o[3].x));  // w8^3 = h(-1 + sign i)
        x[0] = cadd(e[0], o[0]);
        x[4] = csub(e[0], o[0]);
        x[1] = cadd(e[1], o1);
        x[5] = csub(e[1], o1);
        x[2] = cadd(e[2], o2);
        x[6] = csub(e[2], o2);
        x[3] = cadd(e[3], o3);
        x[7] = csub(e[3], o3);
    }
};

// Slot of element p of line l of a tile in shared memory.  Columns (kContig = false) are interleaved,
// p nl + l: consecutive threads take consecutive lines, so a warp touches consecutive banks.  Rows lie
// one after the other, element e = l n + p, in a layout chosen by the stage that writes them so
// that both its writes and the next stage's reads (runs of 16 consecutive elements) spread over
// the 32 banks (a complex value spans two): after the first radix-8 stage (stride-8 writes) the
// low 3 bits of e are XORed with bits 4-6; after the second (runs of 8 at stride 64) every 64
// elements are followed by 8 pad slots; later stages write runs of 16 or more and keep e.
// LOG2W: log2 of the product of the radices before the writing stage.
template <int LOG2N, bool kContig, int LOG2W>
__device__ __forceinline__ int slot(int log2nl, int l, int p) {
    if (!kContig) return (p << log2nl) + l;
    const int e = (l << LOG2N) + p;
    if constexpr (LOG2W == 0) return e ^ ((e >> 4) & 7);
    else if constexpr (LOG2W == 3) return e + 8 * (e >> 6);
    else return e;
}

// Slots of the largest layout (8 pad slots per 64 elements along rows).
template <int LOG2N, bool kContig>
__host__ __device__ __forceinline__ int tile_slots(int nl) {
    return kContig ? (nl << LOG2N) + (nl << LOG2N) / 8 : nl << LOG2N;
}

// Twiddles of the stage after radices L = 2^LOG2L, radix R = 2^LR: w_{LR}^{m j} for m = 1..R-1,
// j = 0..L-1 at tw[(L - 1) + (m - 1) L + j], so that threads with consecutive j read consecutive slots;
// the stages' tables together fill tw[0 .. n-2].
template <int LOG2L, int LR>
__device__ __forceinline__ void stage_twiddles(float2* tw) {
    constexpr int L = 1 << LOG2L, R = 1 << LR;
    for (int e = threadIdx.x; e < (R - 1) * L; e += blockDim.x) {
        const int m = (e >> LOG2L) + 1, j = e & (L - 1);
        float sn, cs;
        sincospif((float)(m * j) * (2.f / (float)(L * R)), &sn, &cs);
        tw[(L - 1) + e] = make_float2(cs, sn);
    }
}

// The tables of all stages: radix-8 stages and, first (kRestFirst) or last, the radix-2 or radix-4 remainder.
template <int LOG2N, bool kRestFirst>
__device__ __forceinline__ void line_twiddles(float2* tw) {
    constexpr int N8 = LOG2N / 3, REST = LOG2N - 3 * N8, B = kRestFirst ? REST : 0;
    if constexpr (REST > 0) stage_twiddles<kRestFirst ? 0 : 3 * N8, REST>(tw);
    if constexpr (N8 >= 1) stage_twiddles<B, 3>(tw);
    if constexpr (N8 >= 2) stage_twiddles<B + 3, 3>(tw);
    if constexpr (N8 >= 3) stage_twiddles<B + 6, 3>(tw);
}

// One Stockham stage of radix R = 2^LR after stages whose radices multiply to L = 2^LOG2L: unit
// (line l, t), t < n/R, j = t mod L, k = t / L, reads a_m = x[t + m n/R], twiddles a_m by
// w_{LR}^{m j}, transforms, writes y[k L R + j + m L], through `load(l, p)` and `put(l, p, v)`; `map(v)` is
// applied to what was loaded, after all loads have been issued (powf between them ran one at a time: the
// x pass of a 512x512x128 grid took 316 us instead of 174).
// kSharedIn, kSharedOut: whether they exchange through the tile in shared memory; a stage that does both
// works in place, so its reads must all come before its writes: it has at most kUnits THREADS units
// (radix 8 and lines_per_block see to that) and a barrier between.
template <int LOG2N, bool kContig, int LR, int LOG2L, int SIGN, int THREADS, bool kSharedIn, bool kSharedOut, class Load,
          class Put, class Map>
__device__ __forceinline__ void stage(int log2nl, const float2* tw, Load&& load, Put&& put, Map&& map) {
    constexpr int R = 1 << LR, LOG2NR = LOG2N - LR, NR = 1 << LOG2NR;
    const int units = 1 << (log2nl + LOG2NR), nl_mask = (1 << log2nl) - 1;
    for (int u0 = 0; u0 < units; u0 += kUnits * THREADS) {
        float2 a[kUnits][R];
#pragma unroll
        for (int q = 0; q < kUnits; ++q) {
            const int u = u0 + q * THREADS + threadIdx.x;
            // consecutive threads: consecutive t along rows, consecutive lines across columns
            const int l = kContig ? u >> LOG2NR : u & nl_mask, t = kContig ? u & (NR - 1) : u >> log2nl;
            if (u < units) {
#pragma unroll
                for (int m = 0; m < R; ++m) a[q][m] = load(l, t + m * NR);
            }
        }
        if (kSharedIn && kSharedOut) __syncthreads();
#pragma unroll
        for (int q = 0; q < kUnits; ++q) {
            const int u = u0 + q * THREADS + threadIdx.x;
            const int l = kContig ? u >> LOG2NR : u & nl_mask, t = kContig ? u & (NR - 1) : u >> log2nl;
            if (u >= units) continue;
            const int j = t & ((1 << LOG2L) - 1), k = t >> LOG2L;
#pragma unroll
            for (int m = 0; m < R; ++m) a[q][m] = map(a[q][m]);
            if constexpr (LOG2L > 0) {
#pragma unroll
                for (int m = 1; m < R; ++m)
                    a[q][m] = cmul<SIGN>(tw[((1 << LOG2L) - 1) + ((m - 1) << LOG2L) + j], a[q][m]);
            }
            Dft<R, SIGN>::run(a[q]);
#pragma unroll
            for (int m = 0; m < R; ++m) put(l, (k << (LOG2L + LR)) + j + (m << LOG2L), a[q][m]);
        }
    }
    // the tile is complete (out), or free for the next writer (in)
    if (kSharedIn || kSharedOut) __syncthreads();
}

struct Same {
    __device__ __forceinline__ float2 operator()(float2 v) const { return v; }
};

// All stages of a tile's lines from `load` to `put`, through x between.  kIn, kOut: whether those ends are x
// itself.  In place, only radix-8 stages: the remainder comes first where the input is not x, else last.
template <int LOG2N, bool kContig, bool kRestFirst, int SIGN, int THREADS, bool kIn, bool kOut, class Load, class Put,
          class Map = Same>
__device__ __forceinline__ void fft_lines(int log2nl, float2* x, const float2* tw, Load&& load, Put&& put,
                                          Map&& map = Map()) {
    constexpr int N8 = LOG2N / 3, REST = LOG2N - 3 * N8, NS = N8 + (REST > 0 ? 1 : 0);
    // radices of the first and the last stage
    constexpr int LF = (kRestFirst && REST > 0) || N8 == 0 ? REST : 3, LE = (!kRestFirst && REST > 0) || N8 == 0 ? REST : 3;
    static_assert(!(kIn && kOut) || REST == 0, "a remainder stage cannot work in place");
    static_assert(!kContig || !kRestFirst, "the row layouts assume radix-8 stages first");
    if constexpr (NS == 1) {
        stage<LOG2N, kContig, LF, 0, SIGN, THREADS, kIn, kOut>(log2nl, tw, load, put, map);
    } else {
        auto out0 = [&](int l, int p, float2 v) { x[slot<LOG2N, kContig, 0>(log2nl, l, p)] = v; };
        auto in0 = [&](int l, int p) { return x[slot<LOG2N, kContig, 0>(log2nl, l, p)]; };
        auto out3 = [&](int l, int p, float2 v) { x[slot<LOG2N, kContig, 3>(log2nl, l, p)] = v; };
        auto in3 = [&](int l, int p) { return x[slot<LOG2N, kContig, 3>(log2nl, l, p)]; };
        auto out6 = [&](int l, int p, float2 v) { x[slot<LOG2N, kContig, 6>(log2nl, l, p)] = v; };
        auto in6 = [&](int l, int p) { return x[slot<LOG2N, kContig, 6>(log2nl, l, p)]; };
        stage<LOG2N, kContig, LF, 0, SIGN, THREADS, kIn, true>(log2nl, tw, load, out0, map);
        if constexpr (NS == 2) {
            stage<LOG2N, kContig, LE, LF, SIGN, THREADS, true, kOut>(log2nl, tw, in0, put, Same());
        } else if constexpr (NS == 3) {
            stage<LOG2N, kContig, 3, LF, SIGN, THREADS, true, true>(log2nl, tw, in0, out3, Same());
            stage<LOG2N, kContig, LE, LF + 3, SIGN, THREADS, true, kOut>(log2nl, tw, in3, put, Same());
        } else {
            stage<LOG2N, kContig, 3, LF, SIGN, THREADS, true, true>(log2nl, tw, in0, out3, Same());
            stage<LOG2N, kContig, 3, LF + 3, SIGN, THREADS, true, true>(log2nl, tw, in3, out6, Same());
            stage<LOG2N, kContig, LE, LF + 6, SIGN, THREADS, true, kOut>(log2nl, tw, in6, put, Same());
        }
    }
}

// What the kernels get; pitches and lengths as in fft_layout.cuh.
struct Plan {
    const float *f, *g;
    float4* ff;
    float2 *z, *a, *b, *c, *d, *e;
    int nx, ny, nz;
    int px, pz, hx, hz, zlen, hlen;
    float kx0, ky0, kz0;  // 2 pi / (n d) per axis
    float norm;           // scale * dV / N
    float power;
    int accumulate;
    int log2nl;           // lines of a tile (of one kind where a kernel takes several)
};

__device__ __forceinline__ float powered(float v, float p) {
    if (p == 1.f) return v;
    return v > 0.f ? powf(v, p) : 0.f;
}

// Wavenumber of index m along an axis of length n (Nyquist -> 0 for the derivative).
__device__ __forceinline__ float wavenumber(int m, int n, float k0) {
    if (2 * m == n) return 0.f;
    return (2 * m < n ? (float)m : (float)(m - n)) * k0;
}

// Block b: rows (b % nbi) nl onwards of plane b / nbi.
template <int LOG2N>
__global__ void __launch_bounds__(kThreads, 4) fft_x_forward_kernel(const Plan P) {
    extern __shared__ __align__(128) unsigned char smraw[];
    float2* const tw = reinterpret_cast<float2*>(smraw);
    float2* const x = tw + (1 << LOG2N);
    line_twiddles<LOG2N, false>(tw);
    __syncthreads();
    const int nbi = P.ny >> P.log2nl, k = blockIdx.x / nbi, j0 = (blockIdx.x % nbi) << P.log2nl;
    const int nodes = (P.ny * P.nz) << LOG2N;
    const int src = (k * P.ny + j0) << LOG2N, dst = k * P.pz + j0 * P.px;
    fft_lines<LOG2N, true, false, -1, kThreads, false, false>(
        P.log2nl, x, tw,
        [&](int l, int p) {
            const int s = checked(src + (l << LOG2N) + p, nodes, kChkFft);
            return make_float2(__ldg(P.f + s), __ldg(P.g + s));
        },
        [&](int l, int p, float2 v) { P.z[checked(dst + l * P.px + p, P.zlen, kChkFft)] = v; },
        [&](float2 v) { return make_float2(powered(v.x, P.power), powered(v.y, P.power)); });
}

// Block b: columns (b % nbi) nl onwards of plane b / nbi.
template <int LOG2N>
__global__ void __launch_bounds__(kThreads, 4) fft_y_forward_kernel(const Plan P) {
    extern __shared__ __align__(128) unsigned char smraw[];
    float2* const tw = reinterpret_cast<float2*>(smraw);
    float2* const x = tw + (1 << LOG2N);
    line_twiddles<LOG2N, false>(tw);
    __syncthreads();
    const int nbi = P.nx >> P.log2nl;
    const int base = (int)(blockIdx.x / nbi) * P.pz + (int)((blockIdx.x % nbi) << P.log2nl);
    auto at = [&](int l, int p) { return checked(base + l + p * P.px, P.zlen, kChkFft); };
    fft_lines<LOG2N, false, false, -1, kThreads, false, false>(
        P.log2nl, x, tw, [&](int l, int p) { return P.z[at(l, p)]; },
        [&](int l, int p, float2 v) { P.z[at(l, p)] = v; });
}

// Block b: columns i = (b % nbi) nl onwards (i <= nx/2) of row j = b / nbi, and their mirrors (-i, -j) as
// lines nl .. 2 nl - 1 of the tile.
template <int LOG2N, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 4 : 2) fft_z_middle_kernel(const Plan P) {
    extern __shared__ __align__(128) unsigned char smraw[];
    constexpr int N = 1 << LOG2N;
    float2* const tw = reinterpret_cast<float2*>(smraw);  // forward, then inverse tables
    float2* const x = tw + 2 * N;
    line_twiddles<LOG2N, true>(tw);
    line_twiddles<LOG2N, false>(tw + N);
    __syncthreads();
    const int nl = 1 << P.log2nl, half = P.nx / 2, nbi = (half >> P.log2nl) + 1;
    const int j = blockIdx.x / nbi, i0 = (blockIdx.x % nbi) << P.log2nl, mj = j == 0 ? 0 : P.ny - j;
    const int log2all = P.log2nl + 1;
    fft_lines<LOG2N, false, true, -1, THREADS, false, true>(
        log2all, x, tw,
        [&](int l, int p) {
            const int i = i0 + (l & (nl - 1));
            if (i > half) return make_float2(0.f, 0.f);
            const int o = l < nl ? j * P.px + i : mj * P.px + (i == 0 ? 0 : P.nx - i);
            return P.z[checked(o + p * P.pz, P.zlen, kChkFft)];
        },
        [&](int l, int p, float2 v) { x[(p << log2all) + l] = v; });
    // the products at p and n - p together: each needs both lines at both
    for (int u = threadIdx.x; u < ((N / 2 + 1) << P.log2nl); u += THREADS) {
        const int l = u & (nl - 1), p = u >> P.log2nl, q = p == 0 ? 0 : N - p;
        float2* const zp = x + (p << log2all) + l;
        float2* const zq = x + (q << log2all) + l;
        const float2 z0 = zp[0], m0 = zq[nl], z1 = zq[0], m1 = zp[nl];
        auto product = [&](float2 zk, float2 zm, int m, float2* out) {
            // F^ = (Z_k + conj Z_-k)/2, G^ = (Z_k - conj Z_-k)/(2i)
            const float2 F = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
            const float2 G = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
            // P = conj(G) F norm, and -i kz P
            const float2 Pk = make_float2(P.norm * fmaf(G.x, F.x, G.y * F.y), P.norm * fmaf(G.x, F.y, -G.y * F.x));
            const float kz = wavenumber(m, N, P.kz0);
            out[0] = Pk;
            out[nl] = make_float2(kz * Pk.y, -kz * Pk.x);
        };
        product(z0, m0, p, zp);
        if (q != p) product(z1, m1, q, zq);
    }
    __syncthreads();
    fft_lines<LOG2N, false, false, 1, THREADS, true, false>(
        log2all, x, tw + N, [&](int l, int p) { return x[(p << log2all) + l]; },
        [&](int l, int p, float2 v) {
            const int i = i0 + (l & (nl - 1));
            if (i > half) return;
            (l < nl ? P.a : P.b)[checked(j * P.hx + i + p * P.hz, P.hlen, kChkFft)] = v;
        });
}

// Block b: kind b % 3 (E and Fy from P, Fz from -i kz P) of columns ((b / 3) % nbi) nl onwards of plane
// (b / 3) / nbi; the kinds that share a source run side by side.
template <int LOG2N>
__global__ void __launch_bounds__(kThreads, 4) fft_y_inverse_kernel(const Plan P) {
    extern __shared__ __align__(128) unsigned char smraw[];
    float2* const tw = reinterpret_cast<float2*>(smraw);
    float2* const x = tw + (1 << LOG2N);
    line_twiddles<LOG2N, false>(tw);
    __syncthreads();
    const int kind = blockIdx.x % 3, b = blockIdx.x / 3, half = P.nx / 2, nbi = (half >> P.log2nl) + 1;
    const int k = b / nbi, i0 = (b % nbi) << P.log2nl;
    const float2* const in = kind == 2 ? P.b : P.a;
    float2* const out = kind == 0 ? P.c : kind == 1 ? P.d : P.e;
    auto at = [&](int l, int p) { return checked(k * P.hz + p * P.hx + i0 + l, P.hlen, kChkFft); };
    fft_lines<LOG2N, false, false, 1, kThreads, false, false>(
        P.log2nl, x, tw,
        [&](int l, int p) {
            if (i0 + l > half) return make_float2(0.f, 0.f);
            const float2 v = in[at(l, p)];
            if (kind != 1) return v;
            const float ky = wavenumber(p, 1 << LOG2N, P.ky0);
            return make_float2(ky * v.y, -ky * v.x);
        },
        [&](int l, int p, float2 v) {
            if (i0 + l <= half) out[at(l, p)] = v;
        });
}

// Block b: rows (b % nbi) nl onwards of plane b / nbi.  y: the finished (E, Fx) rows.
template <int LOG2N>
__global__ void __launch_bounds__(kThreads, 3) fft_x_inverse_kernel(const Plan P) {
    extern __shared__ __align__(128) unsigned char smraw[];
    constexpr int N = 1 << LOG2N;
    float2* const tw = reinterpret_cast<float2*>(smraw);
    float2* const x = tw + N;
    float2* const y = x + tile_slots<LOG2N, true>(1 << P.log2nl);
    line_twiddles<LOG2N, false>(tw);
    __syncthreads();
    const int nbi = P.ny >> P.log2nl, k = blockIdx.x / nbi, j0 = (blockIdx.x % nbi) << P.log2nl;
    const int nodes = (P.ny * P.nz) << LOG2N;
    const int src = k * P.hz + j0 * P.hx, dst = (k * P.ny + j0) << LOG2N;
    // element p of a real row's spectrum from its half; the ends are real
    auto full = [&](const float2* h, int l, int p) {
        const float2 v = h[checked(src + l * P.hx + (2 * p <= N ? p : N - p), P.hlen, kChkFft)];
        return make_float2(v.x, p == 0 || 2 * p == N ? 0.f : 2 * p < N ? v.y : -v.y);
    };
    fft_lines<LOG2N, true, false, 1, kThreads, false, false>(
        P.log2nl, x, tw,
        [&](int l, int p) {
            const float2 v = full(P.c, l, p);
            const float s = 1.f + wavenumber(p, N, P.kx0);  // E^ + i (-i kx E^)
            return make_float2(s * v.x, s * v.y);
        },
        [&](int l, int p, float2 v) { y[(l << LOG2N) + p] = v; });
    __syncthreads();
    fft_lines<LOG2N, true, false, 1, kThreads, false, false>(
        P.log2nl, x, tw,
        [&](int l, int p) {
            const float2 u = full(P.d, l, p), v = full(P.e, l, p);
            return make_float2(u.x - v.y, u.y + v.x);
        },
        [&](int l, int p, float2 v) {
            const float2 u = y[(l << LOG2N) + p];
            float4 o = make_float4(u.y, v.x, v.y, u.x);
            float4* const to = P.ff + checked(dst + (l << LOG2N) + p, nodes, kChkFft);
            if (P.accumulate) {
                const float4 w = *to;
                o = make_float4(w.x + o.x, w.y + o.y, w.z + o.z, w.w + o.w);
            }
            *to = o;
        });
}

int ilog2i(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

// log2 of the lines per tile for lines of n among `avail` neighbours (powers of two): up to `want`, and at
// most what gives `kinds` times as many lines kUnits units of a radix-8 stage per thread.
int lines_per_block(int n, int avail, int want, int threads, int kinds) {
    const int cap = 8 * kUnits * threads / (n * kinds);
    const int L = avail < want ? avail : want;
    return ilog2i(L < cap ? L : cap);
}

template <class K>
cudaError_t launch(K kernel, long long blocks, int threads, size_t values, const Plan& P, cudaStream_t s) {
    const int smem = (int)(values * sizeof(float2));
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kernel<<<(unsigned)blocks, threads, smem, s>>>(P);
    return cudaGetLastError();
}

// f(std::integral_constant<int, log2 n>)
template <class F>
cudaError_t with_log2(int n, F&& f) {
    switch (ilog2i(n)) {
        case 1: return f(std::integral_constant<int, 1>{});
        case 2: return f(std::integral_constant<int, 2>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
        case 9: return f(std::integral_constant<int, 9>{});
        case 10: return f(std::integral_constant<int, 10>{});
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

size_t fft_workspace_bytes(int nx, int ny, int nz) {
    return (size_t)fft_layout(nx, ny, nz).size * sizeof(float2);
}

cudaError_t launch_fft_correlate(const FftLaunch& L, cudaStream_t s) {
    Plan P;
    const FftLayout at = fft_layout(L.nx, L.ny, L.nz);
    P.nx = L.nx; P.ny = L.ny; P.nz = L.nz;
    P.px = at.px; P.pz = at.pz; P.hx = at.hx; P.hz = at.hz;
    P.zlen = at.zlen; P.hlen = at.hlen;
    P.f = L.f;
    P.g = L.g;
    P.ff = L.ff;
    P.z = reinterpret_cast<float2*>(L.ws);
    P.a = P.z + at.a;
    P.b = P.z + at.b;
    P.c = P.z + at.c;
    P.d = P.z + at.d;
    P.e = P.z + at.e;
    P.kx0 = (float)(2.0 * kPi / (L.nx * (double)L.dx));
    P.ky0 = (float)(2.0 * kPi / (L.ny * (double)L.dy));
    P.kz0 = (float)(2.0 * kPi / (L.nz * (double)L.dz));
    P.norm = (float)((double)L.scale * (double)L.dx * L.dy * L.dz / ((double)L.nx * L.ny * L.nz));
    P.power = L.power;
    P.accumulate = L.accumulate;
    const int half = L.nx / 2;
    cudaError_t e;
    P.log2nl = lines_per_block(L.nx, L.ny, kLines, kThreads, 1);
    e = with_log2(L.nx, [&](auto n) {
        constexpr int LN = decltype(n)::value;
        return launch(fft_x_forward_kernel<LN>, (long long)(L.ny >> P.log2nl) * L.nz, kThreads,
                      (size_t)(1 << LN) + tile_slots<LN, true>(1 << P.log2nl), P, s);
    });
    if (e != cudaSuccess) return e;
    P.log2nl = lines_per_block(L.ny, L.nx, kStridedLines, kThreads, 1);
    e = with_log2(L.ny, [&](auto n) {
        constexpr int LN = decltype(n)::value;
        return launch(fft_y_forward_kernel<LN>, (long long)(L.nx >> P.log2nl) * L.nz, kThreads,
                      (size_t)(1 << LN) + tile_slots<LN, false>(1 << P.log2nl), P, s);
    });
    if (e != cudaSuccess) return e;
    e = with_log2(L.nz, [&](auto n) {
        constexpr int LN = decltype(n)::value, T = LN >= 9 ? 512 : 256;
        P.log2nl = lines_per_block(L.nz, half, kStridedLines / 2, T, 2);
        return launch(fft_z_middle_kernel<LN, T>, (long long)((half >> P.log2nl) + 1) * L.ny, T,
                      (size_t)(2 << LN) + tile_slots<LN, false>(2 << P.log2nl), P, s);
    });
    if (e != cudaSuccess) return e;
    P.log2nl = lines_per_block(L.ny, half, kStridedLines, kThreads, 1);
    e = with_log2(L.ny, [&](auto n) {
        constexpr int LN = decltype(n)::value;
        return launch(fft_y_inverse_kernel<LN>, 3LL * ((half >> P.log2nl) + 1) * L.nz, kThreads,
                      (size_t)(1 << LN) + tile_slots<LN, false>(1 << P.log2nl), P, s);
    });
    if (e != cudaSuccess) return e;
    P.log2nl = lines_per_block(L.nx, L.ny, kLines, kThreads, 1);
    return with_log2(L.nx, [&](auto n) {
        constexpr int LN = decltype(n)::value;
        return launch(fft_x_inverse_kernel<LN>, (long long)(L.ny >> P.log2nl) * L.nz, kThreads,
                      (size_t)(1 << LN) + tile_slots<LN, true>(1 << P.log2nl) + ((size_t)1 << (LN + P.log2nl)), P, s);
    });
}

PP_CHECK_READER(check_flags_fft)

}  // namespace pp
