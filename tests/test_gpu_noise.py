"""fc_noise (App. A perturbation) on the GPU vs the FP64 oracle, through the C ABI."""
import math

import numpy as np
import pytest

from oracle import noise
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2002_01392_gb300 import api as a
    assert torch.cuda.is_available()
    return a


def _run(api, Nx, Ny, Nz, dtype, seed, **kw):
    p = api.noise_params(**kw)
    cnt = api.noise_modes(p)
    draws = synth.noise_draws(cnt, seed)
    out = torch.full((3, Nz, Ny, Nx), float("nan"), dtype=dtype, device="cuda")
    api.fc_noise(p, draws, out)
    torch.cuda.synchronize()
    return out.cpu().double().numpy(), draws


def _oracle(Nx, Ny, Nz, draws, **kw):
    d = noise.DEFAULTS
    return noise.noise_field(Nx, Ny, Nz, draws, kw.get("Lx", d["Lx"]), kw.get("Ly", d["Ly"]), kw.get("Lz", 1.0),
                             (kw.get("kperp2_min", 4.0), kw.get("kperp2_max", 25.0)),
                             (kw.get("m_min", 2), kw.get("m_max", 5)), (kw.get("slope_phi", -4.0),
                                                                        kw.get("slope_psi", -3.0)),
                             kw.get("amplitude", 1.0))


@pytest.mark.parametrize("Nx,Ny,Nz,kw", [
    (16, 16, 33, {}),
    (13, 11, 20, {}),                                                    # odd sizes, smallest resolving grid
    (24, 14, 21, {"Lx": 4 * math.pi, "Lz": 2.0, "amplitude": 0.3}),
    (18, 20, 40, {"Ly": 3.0, "kperp2_min": 1.0, "kperp2_max": 9.0, "m_min": 1, "m_max": 3,
                  "slope_phi": -2.0, "slope_psi": -1.5}),
])
def test_noise_float64_matches_oracle(api, Nx, Ny, Nz, kw):
    out, draws = _run(api, Nx, Ny, Nz, torch.float64, 11, **kw)
    ref = _oracle(Nx, Ny, Nz, draws, **kw)
    amp = kw.get("amplitude", 1.0)
    assert np.abs(out - ref).max() < 1e-13 * amp
    assert np.abs(out[:, [0, -1]]).max() < 1e-14 * amp        # no slip at both walls
    assert abs(np.abs(out).max() - amp) < 1e-15 * amp


def test_noise_float32_matches_oracle(api):
    out, draws = _run(api, 32, 32, 65, torch.float32, 12)
    ref = _oracle(32, 32, 65, draws)
    # two float32 roundings of values <= 1 (synthesis, scaling) and the float32 maximum
    assert np.abs(out - ref).max() < 3e-7
    assert np.abs(out[:, [0, -1]]).max() < 1e-7


def test_noise_full_size_sampled(api):
    """1024^2 x 513 float32 (the Boussinesq grid of the RK-step workload):
    every 64th x and y column against the oracle on the 16 x 16 x 513 grid
    that holds exactly those points, up to the one global scale (the maximum
    is taken over different point sets), which the largest magnitude fixes."""
    Nx = Ny = 1024
    Nz = 513
    p = api.noise_params()
    draws = synth.noise_draws(api.noise_modes(p), 13)
    out = torch.empty((3, Nz, Ny, Nx), dtype=torch.float32, device="cuda")
    api.fc_noise(p, draws, out)
    torch.cuda.synchronize()
    assert abs(out.abs().max().item() - 1.0) < 1.2e-7
    assert out[:, [0, -1]].abs().max().item() < 1e-7
    assert torch.isfinite(out).all().item()
    sample = out[:, :, ::64, ::64].cpu().double().numpy()
    ref = _oracle(16, 16, Nz, draws)
    c = float((sample * ref).sum() / (ref * ref).sum())
    assert 0.5 < c <= 1.0 + 1e-6
    assert np.abs(sample - c * ref).max() < 3e-7
    del out
    torch.cuda.empty_cache()


@pytest.mark.parametrize("Nx,Ny,Nz,kw", [
    (11, 11, 4, {}),                        # two points per sum, smallest grid
    (12, 12, 5, {}),                        # four points per sum, smallest grid
    (14, 9 + 8, 5, {"kperp2_max": 10.0}),   # Nx even, not a multiple of four; a short last row group
    (128, 13, 9, {}),
    (516, 12, 3, {}),                       # more points than threads
    (204, 203, 3, {"kperp2_min": 9999.0, "kperp2_max": 10001.0, "m_min": 1, "m_max": 1}),   # fewer rows per block
])
def test_noise_folded_rows_match_oracle(api, Nx, Ny, Nz, kw):
    """The folded row sums in both arithmetics, one value at a time."""
    out64, draws = _run(api, Nx, Ny, Nz, torch.float64, 17, **kw)
    out32, _ = _run(api, Nx, Ny, Nz, torch.float32, 17, **kw)
    ref = _oracle(Nx, Ny, Nz, draws, **kw)
    assert np.abs(out64 - ref).max() < 1e-13
    # one float32 rounding of values <= 1; the pairs' own error is below 1e-12
    assert np.abs(out32 - ref).max() <= 2.0 ** -24 + 1e-12


@pytest.mark.parametrize("size,amplitude", [(1e-18, 1e-25), (1e18, 1e25), (1e-12, 1e30), (1.0, 2e-38), (1.0, 3e38)])
def test_noise_box_sizes_and_amplitudes(api, size, amplitude):
    """Boxes and amplitudes whose ratio to the unscaled sums leaves float's range: float32 output is the float64 one,
    rounded (2^-24 of a value, 2^-150 where it is subnormal, each twice for the shift)."""
    kw = {"Lx": 2 * np.pi * size, "Ly": 2 * np.pi * size, "Lz": size, "kperp2_min": 4.0 / size ** 2,
          "kperp2_max": 25.0 / size ** 2, "amplitude": amplitude}
    out64, _ = _run(api, 14, 12, 9, torch.float64, 5, **kw)
    out32, _ = _run(api, 14, 12, 9, torch.float32, 5, **kw)
    assert abs(np.abs(out64).max() / amplitude - 1) < 1e-14
    assert np.abs(out32 - out64).max() <= 2.0 ** -23 * amplitude + 2.0 ** -149
