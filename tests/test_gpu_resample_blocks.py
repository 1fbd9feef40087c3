"""Resampling at the limits of its passes: chunks of one to 512 scores and longer (streamed),
draws below, at and above a pass of 512, scores with NaN and -inf, flat scores (every chunk
weighs the same), against the inverse CDF in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 512, 513, 1025, 262145, 524288, 524289, 700001])
@pytest.mark.parametrize("m", [1, 16, 512, 513, 1300])
def test_draws_at_pass_limits(orc, n, m):
    """Draws equal the oracle's wherever its CDF margin exceeds 1e-5 (the FP32 bound of the
    resampling tests); log normaliser within 1e-5 relative."""
    from paper_2312_08715_gb300 import b3d
    rng = np.random.default_rng(n + m)
    ll = (rng.uniform(-8.0, 0.0, size=n) if n % 2 else np.full(n, -3.0)).astype(np.float32)
    ll[rng.random(n) < 0.1] = -np.inf
    ll[n // 2] = 0.0
    clean = ll.astype(np.float64)
    if n > 100:
        ll[n // 3] = np.nan  # weighs nothing
        clean[n // 3] = -np.inf
    ctx = b3d.Context(0)
    logz, idx, logq = ctx.lse_resample(torch.as_tensor(ll, device="cuda"), m, 77, 2)
    ctx.sync()
    Z, _ = orc.lse(clean)
    assert abs(float(logz[0]) - Z) <= 1e-5 * max(1.0, abs(Z)) + 1e-4
    oi, oq, margin = orc.resample(clean, m, 77, 2)
    got, solid = idx.cpu().numpy(), margin > 1e-5
    np.testing.assert_array_equal(got[solid], oi[solid])
    assert np.isfinite(ll[got]).all()
    np.testing.assert_allclose(logq.cpu().numpy(), ll[got].astype(np.float64) - Z, atol=2e-4 * max(1.0, abs(Z)))
    ctx.close()
