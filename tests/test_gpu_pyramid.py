"""The pyramid's normalised levels (read back as the network's input pairs, level
257^2) against FP64, at frame sides on both sides of the statistics kernel's
one-sweep limit (1024 columns) and with zero to four restrictions above the
level."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("side", [256, 512, 1024, 2048, 4096])
def test_normalised_level_matches_fp64(syn, side, storage):
    """FP32 restriction adds at most four roundings per level, the normalisation
    and storage one each: (4 k + 2) 2^-24 of the largest value after k
    restrictions, or the BF16 storage's half unit (2^-8) of each value."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1712_02533_gb300 import _build
    _build.build()
    import paper_1712_02533_gb300 as reg
    rng = np.random.default_rng(side)
    y = np.arange(side) / side
    fr = (300.0 + 40.0 * np.sin(9.0 * y)[:, None] * np.cos(7.0 * y)[None, :]
          + rng.poisson(20.0, size=(3, side, side))).astype(np.float32)
    k = int(np.log2(side)) - 8
    x = torch.empty((2, 2, 256, 256), device="cuda")
    with reg.Series(fr, reg.default_params(n_levels=k + 1, storage=storage)) as s:
        s.cnn_pairs(0, 2, x)
    got = x.cpu().numpy()
    for f in range(3):
        v = np.pad(fr[f].astype(np.float64), ((0, 1), (0, 1)), mode="edge")
        for _ in range(k):
            p = np.pad(v, 1, mode="reflect")
            p = 0.25 * p[:-2:2] + 0.5 * p[1:-1:2] + 0.25 * p[2::2]
            v = 0.25 * p[:, :-2:2] + 0.5 * p[:, 1:-1:2] + 0.25 * p[:, 2::2]
        h2 = 1.0 / (v.shape[0] - 1) ** 2
        a, b, c, d = v[:-1, :-1], v[:-1, 1:], v[1:, 1:], v[1:, :-1]
        v = v - h2 * 0.25 * (a + b + c + d).sum()
        a, b, c, d = v[:-1, :-1], v[:-1, 1:], v[1:, 1:], v[1:, :-1]
        q = 4 * (a * a + b * b + c * c + d * d) + 4 * (a * b + b * c + c * d + d * a) + 2 * (a * c + b * d)
        sig = np.sqrt(h2 * q.sum() / 36.0)
        # the raw values' rounding (their mean is far from zero) over sigma
        tol = (4 * k + 2) * 2.0 ** -24 * np.abs(fr[f]).max() / sig
        want = (v / sig)[:256, :256]
        bound = tol + (np.abs(want) * 2.0 ** -8 if storage else 0.0)
        for g in ([got[f, 0]] if f < 2 else []) + ([got[f - 1, 1]] if f > 0 else []):
            assert (np.abs(g - want) <= bound).all(), (side, f, np.abs(g - want).max())
