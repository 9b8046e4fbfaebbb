"""fd_forward_noalloc on every copy width its step kernel has (rows and buffers
aligned to 16, 8 and 4 bytes), on extents at and around its 32x16 tiles and
x-chunks, thinner than the stencil, and without a damping field, against the
FP64 oracle (FP32 parity bound 1e-5 of the larger of the two levels' norms)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1912_00695_gb300 import _abi, inputs

pytestmark = pytest.mark.gpu

CASES = [
    # shape, space order, element offset of the buffers, damping, steps
    ((40, 33, 64), 8, 0, True, 25),   # 16-byte rows and buffers
    ((40, 33, 64), 8, 2, True, 25),   # 16-byte rows, buffers at 8 bytes
    ((40, 33, 64), 8, 1, True, 25),   # ... at 4 bytes
    ((37, 31, 66), 4, 0, True, 30),   # 8-byte rows, a 2-point tail
    ((37, 47, 65), 16, 0, True, 20),  # 4-byte rows, a 1-point tail
    ((9, 16, 32), 2, 0, False, 30),   # one tile, no damping field
    ((17, 49, 35), 12, 0, False, 20),
    ((3, 2, 5), 14, 0, True, 20),     # thinner than the stencil on every axis
    ((1, 17, 33), 6, 0, True, 20),
    ((70, 5, 3), 10, 3, True, 20),
]


@pytest.mark.parametrize("shape,k,off,damped,nt", CASES)
def test_noalloc_widths_and_edges(oracle_mod, shape, k, off, damped, nt):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    m = (1.0 / rng.uniform(1500.0, 4500.0, size=shape) ** 2).astype(np.float32)
    eta = (m * rng.uniform(0.0, 40.0, size=shape) * (rng.random(shape) < 0.5)).astype(np.float32)
    dt = 0.85 * oracle_mod.dt_max(k, inputs.H, 4500.0)
    nodes = [(shape[0] // 2, shape[1] // 2, shape[2] // 2), (0, shape[1] - 1, shape[2] - 1)]
    wav = np.stack([inputs.ricker(25.0, dt, nt), inputs.ricker(18.0, dt, nt, amplitude=2.0)])
    u0, u1 = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))

    def buf(a):  # the array at an offset of `off` floats from an aligned address
        v = torch.zeros(a.size + 8, dtype=torch.float32, device="cuda")[off:off + a.size]
        v.copy_(torch.from_numpy(a).reshape(-1))
        return v

    d_u, d_up, d_m, d_eta = buf(u0), buf(u1), buf(m), buf(eta)
    d_wav = torch.from_numpy(wav).cuda()
    amax = _abi.fd_forward_noalloc(d_u, d_up, d_m, d_eta if damped else None, shape, k, inputs.H, dt, nodes, d_wav,
                                   nt, step0=0, nt=nt, stream=torch.cuda.current_stream().cuda_stream)
    new, old = (d_u, d_up) if nt % 2 == 0 else (d_up, d_u)
    got = [x.cpu().numpy().reshape(shape) for x in (new, old)]
    want = oracle_mod.forward(m.astype(np.float64), eta.astype(np.float64) if damped else None, k, inputs.H, dt, nt,
                              nodes, wav.astype(np.float64), u0=u0.astype(np.float64), u_prev0=u1.astype(np.float64),
                              step0=0)
    scale = max(np.linalg.norm(w) for w in want[:2])
    for g, w in zip(got, want):
        assert np.linalg.norm(g - w) <= 1e-5 * scale
    assert np.isfinite(amax) and amax >= np.abs(got[0]).max()
