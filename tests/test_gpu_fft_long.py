"""All four components of the FFT path on long axes, and the largest grid it accepts.

Bar: that of the other FFT tests, 2e-5, of the largest magnitude of the pair of components that one complex
transform carries as its real and imaginary parts, (E, Fx) and (Fy, Fz): rounding is relative to the transform's
values, whichever part they lie in."""
import numpy as np
import pytest
import torch

from paper_2401_14564_gb300 import pp
from test_gpu_fft import TOL, fields, grid, run

pytestmark = pytest.mark.gpu


def correlation64(f, tip, g, scale, power):
    """(Fx, Fy, Fz, E) by numpy's FFT in 64 bits, the gradient spectral with the Nyquist terms dropped."""
    a, b = (np.clip(np.asarray(v, np.float32).astype(np.float64), 0.0, None) ** power for v in (f, tip))
    S = np.conj(np.fft.fftn(b)) * np.fft.fftn(a) * scale * g["dx"] * g["dy"] * g["dz"]
    out = np.empty(f.shape + (4,))
    out[..., 3] = np.fft.ifftn(S).real
    for c, (n, d) in enumerate((("nx", "dx"), ("ny", "dy"), ("nz", "dz"))):
        k = 2.0 * np.pi * np.fft.fftfreq(g[n], g[d])
        k[g[n] // 2] = 0.0
        out[..., c] = np.fft.ifftn(-1j * k.reshape([-1 if a == 2 - c else 1 for a in range(3)]) * S).real
    return out


@pytest.mark.parametrize("shape", [(256, 4, 8), (512, 8, 4), (1024, 4, 8), (4, 256, 8), (8, 512, 4), (4, 1024, 8),
                                   (8, 4, 256), (4, 8, 512), (8, 4, 1024), (64, 512, 16), (512, 16, 64), (16, 64, 512)])
def test_forces_on_long_axes_match_64_bits(shape):
    g = grid(*shape, d=(0.05, 0.07, 0.06))
    f, tip = fields(g, sum(shape))
    got, ref = run(f, tip, g, scale=1.3, power=1.05), correlation64(f, tip, g, 1.3, float(np.float32(1.05)))
    for pair in ((3, 0), (1, 2)):
        off = np.abs(got[..., pair] - ref[..., pair]).max()
        assert off <= TOL * np.abs(ref[..., pair]).max(), (pair, off)


def test_the_largest_grid_against_the_closed_form():
    # plane waves on both sides, of the same wavevectors: F^ and G^ are large at the same coefficients (the two
    # real transforms run as one complex one, so each rounds at the larger's scale), and the correlation is known,
    # sum_h g[h] f[n + h] = N/2 sum_w A_w B_w cos(k_w n + phi_w - psi_w)
    n, d, scale = 1024, 0.1, 0.7
    if torch.cuda.mem_get_info()[0] < 70 << 30:
        pytest.skip("needs 60 GB")
    gr = pp.make_grid(grid(n, n, n, d=(d, d, d)), 0)
    waves = [(1.0, 0.9, n // 8, n // 32, n // 16, 0.3, 1.0), (0.6, 1.1, n // 32, n // 4, n // 8, 1.1, -0.4),
             (0.8, 0.7, -n // 16, n // 8, n // 4, 2.0, 0.2)]
    i = torch.arange(n, device="cuda", dtype=torch.float64)

    def angle(k, a, b, c):
        return 2.0 * np.pi / n * (((a * i)[None, :] + (b * i)[:, None] + c * k) % n)

    f, tip = (torch.empty((n, n, n), device="cuda") for _ in range(2))
    for k in range(n):
        f[k] = sum(A * torch.cos(angle(k, a, b, c) + phi) for A, B, a, b, c, phi, psi in waves)
        tip[k] = sum(B * torch.cos(angle(k, a, b, c) + psi) for A, B, a, b, c, phi, psi in waves)
    ff = torch.full((pp.pp_ff_floats(gr),), float("nan"), device="cuda")
    ws = torch.empty(pp.pp_fft_workspace(gr) // 4, device="cuda")
    pp.pp_fft_correlate(f.view(-1), tip.view(-1), gr, scale, 1.0, ff, ws)
    torch.cuda.synchronize()
    got = ff.view(n, n, n, 4)
    norm = scale * float(np.float32(d)) ** 3 * 0.5 * n ** 3
    worst, largest = torch.zeros(2, device="cuda", dtype=torch.float64), torch.zeros(2, device="cuda", dtype=torch.float64)
    for k in range(n):
        ref = torch.zeros((n, n, 4), device="cuda", dtype=torch.float64)
        for A, B, a, b, c, phi, psi in waves:
            t = angle(k, a, b, c) + phi - psi
            ref[..., 3] += A * B * torch.cos(t)
            for q, m in enumerate((a, b, c)):
                ref[..., q] += A * B * 2.0 * np.pi * m / (n * d) * torch.sin(t)
        off = (got[k].double() / norm - ref).abs().amax((0, 1))
        top = ref.abs().amax((0, 1))
        worst = torch.maximum(worst, torch.stack([off[[3, 0]].max(), off[[1, 2]].max()]))
        largest = torch.maximum(largest, torch.stack([top[[3, 0]].max(), top[[1, 2]].max()]))
    assert (worst <= TOL * largest).all(), (worst / largest).tolist()
