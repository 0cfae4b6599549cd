"""Host-side checks of the noise-parameter calls (no GPU: the plan's library handle is
never reached, or is replaced by a recorder)."""

from __future__ import annotations

import numpy as np
import pytest


def _bare_plan(n_filters, n_lags):
    import paper_0906_1775_gb300 as mm
    plan = mm.Plan.__new__(mm.Plan)
    plan._h = None
    plan.stats = {"n_filters": n_filters, "n_lags": n_lags}
    return plan


@pytest.mark.parametrize("n_lags", [64, 100])          # formed on the device, on the host
@pytest.mark.parametrize("shape", [(1, 64), (2, 63), (2, 128), (127,), (0, 64)])
def test_noise_vjp_refuses_lag_gradients_of_another_size(n_lags, shape):
    """The device route reads n_filters x n_lags values from the pointer it is given."""
    import torch
    plan = _bare_plan(2, n_lags)
    prm = np.array([[1.0, 0.1, 1.5], [0.9, 0.2, 1.2]])
    with pytest.raises(ValueError, match="grad_lags"):
        plan.noise_vjp(100.0, prm, torch.zeros(shape, dtype=torch.float64))
