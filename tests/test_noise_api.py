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


def test_parameter_rows_beyond_the_filters_are_ignored():
    """MadmapSolve with one parameter row per detector of a larger set: a plan over the
    first of them takes its own rows; fewer rows than filters are refused."""
    import torch
    import paper_0906_1775_gb300 as mm

    class Recorder:
        stats = {"n_filters": 2, "n_lags": 64}
        seen = []

        def set_noise(self, fs, params):
            if params.shape != (2, 3):
                raise ValueError("params must be [n_filters, 3]")
            self.seen.append((fs, params))

        def solve(self, d, **kw):
            return torch.zeros((1, 1), dtype=torch.float64), {}

    prm = torch.arange(1.0, 10.0, dtype=torch.float64).reshape(3, 3)
    plan = Recorder()
    mm.MadmapSolve.apply(torch.zeros(4), prm, plan, 50.0, None)
    assert plan.seen[0][0] == 50.0 and np.array_equal(plan.seen[0][1], prm[:2].numpy())
    with pytest.raises(ValueError):
        mm.MadmapSolve.apply(torch.zeros(4), prm[:1], plan, 50.0, None)
