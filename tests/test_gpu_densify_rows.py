"""The row copies of the densification step (SH rows and carried arrays) for
row widths around the vector and block sizes, and its decisions at thresholds
that float32 cannot tell apart from the quotient."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _scene(n, sh, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    k = (sh + 1) ** 2
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)
    return dict(means=r(n, 3), log_scales=r(n, 3) - 3.0, quats=r(n, 4), opacity_logits=r(n), sh=r(n, k, 3)), g


@pytest.mark.parametrize("n", [1, 85, 86, 5000])
@pytest.mark.parametrize("sh,widths", [(0, (1, 3)), (1, (4, 5)), (2, (7, 48)), (3, (50, 4095)), (3, (4096, 4100)), (0, (9001,))])
def test_rows_follow_their_source(cuda_lib, n, sh, widths):
    if n > 100 and max(widths) > 4000:
        n = 100
    p, g = _scene(n, sh, n + sh)
    e1, e2 = (torch.rand(n, device="cuda", generator=g) for _ in range(2))
    den = torch.randint(0, 4, (n,), device="cuda", generator=g).float()
    z = torch.randn(n, 2, 3, device="cuda", generator=g)
    carry = [torch.randn(n, w, device="cuda", generator=g) for w in widths]
    new, src, kind, moved = cuda_lib.densify(p, sh, e1, e2, den, z, 0.3, 0.3, -0.8, -3.0, carry=carry)
    assert torch.equal(new["sh"], p["sh"][src]) and torch.equal(new["quats"], p["quats"][src])
    for m, c in zip(moved, carry):
        assert torch.equal(m, torch.where((kind == 0)[:, None], c[src], torch.zeros_like(m)))


@pytest.mark.parametrize("threshold", [2e-4, 0.0, -1.0, 1e-40, 3e-39, 1e39, 0.1])
def test_decisions_at_the_threshold(cuda_lib, threshold):
    n = 4096
    rng = np.random.default_rng(8)
    den = rng.integers(0, 9, n).astype(np.float32)
    with np.errstate(over="ignore"):
        e = (den.astype(np.float64) * threshold).astype(np.float32)
        for _ in range(2):  # a few units in the last place around the threshold
            e = np.nextafter(e, np.where(rng.random(n) < 0.5, np.float32(np.inf), -np.float32(np.inf)))
    e[::17], e[5::17], e[9::17] = 0.0, np.float32(np.nan), np.float32(3e38)
    p, _ = _scene(n, 0, 1)
    p["log_scales"].fill_(0.0)
    p["opacity_logits"].fill_(2.0)
    t = lambda a: torch.tensor(a, device="cuda")
    _, src, _, _ = cuda_lib.densify(p, 0, t(e), t(e), t(den), torch.zeros(n, 2, 3, device="cuda"), threshold, threshold,
                                    -9.0, -1.0)
    d = den.astype(np.float64)
    with np.errstate(all="ignore"):
        mean = np.where(d > 0, e.astype(np.float64) / d, 0.0)
        split = mean >= threshold
    np.testing.assert_array_equal(np.bincount(src.cpu().numpy(), minlength=n), np.where(split, 2, 1))
