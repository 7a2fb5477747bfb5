// Layout of the FFT path's scratch (fft.cu), host side and without CUDA, so that it can be checked for every
// accepted size without a GPU (tests/test_fft_layout_cpu.py).
//
// The full spectrum z holds node (i, j, k) at k pz + j px + i with px = nx + 16 and pz = px ny + 16; a half
// spectrum (i <= nx/2) at k hz + j hx + i.  The y and z strides are then not powers of two (a power-of-two stride
// sends every row of a pass to the same memory channels).  Of the room of three full arrays, z has the first
// and the half arrays a = P and b = -i kz P the end; once z is spent, c = E, d = Fy and e = Fz along x take its
// place and the gap (5 halves fit 3 wholes).
#pragma once

#include <cstdint>

namespace pp {

struct FftLayout {
    int px, pz, hx, hz;
    int zlen, hlen;               // values of z and of a half array: 1040 x 1024 + 16 times 1024 at most, so
                                  // offsets inside one array fit 32 bits; where the arrays start does not
    int64_t a, b, c, d, e, size;  // first value of each half array, and values in all
};

inline FftLayout fft_layout(int nx, int ny, int nz) {
    FftLayout L;
    L.px = nx + 16;
    L.pz = L.px * ny + 16;
    // (below 64 nodes along x the narrower pitch keeps five halves inside three wholes)
    L.hx = nx / 2 + (nx >= 64 ? 16 : 2);
    L.hz = L.hx * ny + 8;
    L.zlen = L.pz * nz;
    L.hlen = L.hz * nz;
    L.size = 3 * (int64_t)L.zlen;
    L.a = L.size - 2 * (int64_t)L.hlen;
    L.b = L.a + L.hlen;
    L.c = 0;
    L.d = L.hlen;
    L.e = 2 * (int64_t)L.hlen;
    return L;
}

}  // namespace pp
