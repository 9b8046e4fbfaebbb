"""fd_forward_noalloc and a handle's expanded form hold the same per-point
arithmetic in two kernels: from the same state, on the same model, damping and
source, they give the same bits (h = 8 and dt a few significant bits, so that both
round the coefficients alike), at every copy width of the caller's rows."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1912_00695_gb300 as fd
from paper_1912_00695_gb300 import _abi, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interior,nbl,k", [((30, 25, 44), 6, 2), ((41, 38, 50), 8, 8), ((35, 30, 33), 4, 12),
                                            ((50, 44, 61), 5, 16)])
@pytest.mark.parametrize("damped", [True, False])
def test_same_bits_as_a_handle(interior, nbl, k, damped):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(k)
    shape = tuple(n + 2 * nbl for n in interior)
    h, dt, nt = 8.0, 0.75 * 2.0 ** -10, 21
    m = (1.0 / rng.uniform(1500.0, 4000.0, size=shape) ** 2).astype(np.float32)
    eta = np.zeros(shape, dtype=np.float32)
    if damped:
        eta[...] = m * rng.uniform(0.0, 40.0, size=shape) * (rng.random(shape) < 0.5)
    wav = inputs.ricker(25.0, dt, nt)
    u0, u1 = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    src = tuple(n // 3 for n in interior)
    with fd.Shot(interior, k, h, dt, nbl, form="expanded", kernel="tma") as shot:
        shot.set_model(m, eta)
        shot.inject(*src, wav)
        shot.load_state(u0, u1, 0)
        shot.forward(nt)
        want = shot.wavefield(0), shot.wavefield(1)
    d = [torch.from_numpy(a).cuda() for a in (u0, u1, m, eta)]
    d_wav = torch.from_numpy(wav).cuda()
    _abi.fd_forward_noalloc(d[0], d[1], d[2], d[3] if damped else None, shape, k, h, dt, [tuple(c + nbl for c in src)],
                            d_wav, nt, step0=0, nt=nt, stream=torch.cuda.current_stream().cuda_stream)
    got = (d[1], d[0]) if nt % 2 else (d[0], d[1])
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g.cpu().numpy(), w)
