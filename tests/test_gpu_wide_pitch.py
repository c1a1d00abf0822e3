"""The allocation-free step on thin domains in arrays of a very wide row pitch: the bits of a tight pitch.

The pitch is the caller's, up to 524288 / Ny elements; chunks of 9, 17 and 33 values, rows that bulk copies move and
rows that they cannot (pitch no multiple of four).  Columns past Nx belong to the caller and keep their values.
"""
import numpy as np
import pytest

from gpu_helpers import need_gpu
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,p,pitches", [(24, 2, 2, (131072, 131071, 60000)), (24, 5, 3, (65536, 65535, 16384)),
                                             (300, 6, 2, (65536, 16384)), (1500, 7, 1, (65536, 65533)),
                                             (4000, 6, 2, (65536, 65535)), (40, 28, 2, (17000, 4099))])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_wide_pitch_keeps_the_bits(nx, ny, p, pitches, scheme):
    wf = need_gpu()
    import torch

    Lx, Ly, Nx, Ny = nx * H_ELEMENT, ny * H_ELEMENT, nx + p, ny + p
    x, y = greville(nx, p, Lx), greville(ny, p, Ly)
    T0 = 300.0 + 700.0 * np.exp(-((x[None, :] - 0.4 * Lx) ** 2 + (y[:, None] - 0.5 * Ly) ** 2) / 18.0)
    f0 = np.random.RandomState(nx + p).uniform(0.0, 1.0, T0.shape)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=1.2, wind_y=-0.7, precision=wf.WF_FP32,
                               scheme=wf.WF_PR if scheme == "pr" else wf.WF_STRANG_CN)
    sim = wf.Simulation(nx, ny, p, 1e-3, prm)
    out = []
    for pitch in (Nx, *pitches):
        a = [torch.full((Ny, pitch), -7.0, dtype=torch.float32, device="cuda") for _ in range(2)]
        for t, t0 in zip(a, (T0, f0)):
            t[:, :Nx] = torch.from_numpy(t0.astype(np.float32))
        torch.cuda.synchronize()
        assert wf.wf_step_noalloc(sim.h, a[0].data_ptr(), a[1].data_ptr(), pitch, 2) == wf.WF_OK
        assert sim.sync() == wf.WF_OK
        assert all(bool((t[:, Nx:] == -7.0).all()) for t in a), pitch
        out.append([t[:, :Nx].cpu().numpy().copy() for t in a])
    sim.close()
    assert np.isfinite(out[0][0]).all() and not np.array_equal(out[0][0], T0.astype(np.float32))
    for pitch, o in zip(pitches, out[1:]):
        assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1]), pitch
