"""The net's input features where a plane holds values of widely different sizes: each voxel against its own terms, not
against the plane's largest value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1508_07982_gb300 import lbm as mod
    return mod


@pytest.mark.parametrize("level", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("decay", [0, 3, 5, 6, 12, 40])
def test_every_voxel_keeps_the_bits_of_its_own_terms(lbm, level, decay):
    """Velocities that fall by 2^-decay from cell to cell, along x, along y and along both, with both signs (terms that
    cancel), over the planes that hold the largest as well.  FP64 products and sums of the eight terms, a rounding of
    the weight with the scale included, are off by at most 16 x 2^-53 of the sum of the terms' sizes; FP32 rounds the
    result."""
    import torch
    B, halo = 8, 2
    rng = np.random.default_rng(100 * level + decay)
    r = np.arange(B)
    fall = [np.ldexp(1.0, -decay * r)[None, None, :], np.ldexp(1.0, -decay * r)[None, :, None]]
    noise = rng.uniform(0.5, 1.0, (4, B, B, B)) * rng.choice([-1.0, 1.0], (4, B, B, B))
    rho = 1.0 + 0.01 * noise[0]
    u = 0.1 * np.stack([noise[1] * fall[0], noise[2] * fall[1], noise[3] * fall[0] * fall[1]])
    u[0, :, 2] = 0.0                      # zeros among them
    blocks = np.array([[0, 0, 0], [(1 << level) - 1] * 3], np.int32)
    t = lambda a: torch.tensor(a, device="cuda")
    _, skip = lbm.warmstart_features(t(rho.reshape(-1)), t(u.reshape(3, -1)), np.array([1, 1, 1], np.int32), B, 0, level,
                                     halo, t(blocks), None, 100.0, 25.0)
    skip = skip.cpu().numpy()
    D, s = B + 2 * halo, 0.5 ** level
    for k in range(2):
        p = [(blocks[k, a] * B - halo + np.arange(D) + 0.5) * s for a in range(3)]
        lo = [np.floor(v - 0.5).astype(int) for v in p]
        w = [(v - 0.5 - f).astype(np.longdouble) for v, f in zip(p, lo)]
        for c, f in enumerate([rho - 1.0, *u]):
            val, size = np.zeros((D, D, D), np.longdouble), np.zeros((D, D, D), np.longdouble)
            for corner in range(8):
                d = [corner & 1, (corner >> 1) & 1, corner >> 2]
                idx = [np.clip(lo[a] + d[a], 0, B - 1) for a in range(3)]
                ww = [w[a] if d[a] else 1 - w[a] for a in range(3)]
                term = (ww[2][:, None, None] * ww[1][None, :, None] * ww[0][None, None, :]) * f[np.ix_(idx[2], idx[1], idx[0])]
                val += term
                size += np.abs(term)
            scale = 100.0 if c == 0 else 25.0
            err = np.abs(skip[k, ..., c] - val * scale)
            bound = 2.0 ** -24 * np.abs(val * scale) + 2.0 ** -49 * size * scale + 2.0 ** -149
            assert (err <= bound).all(), (c, float((err / bound).max()))
