"""Rows that the last tile of the training kernel lacks."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NF, NH = 16, 64
W1, B1, W2, B2 = 0, NF * NH, NF * NH + NH, NF * NH + NH + NH * NH


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16])
def test_missing_rows_add_nothing(n):
    """An infinite weight behind a unit that no sample activates: the unit it
    feeds is dead (0 * inf), and the gradient is that of a finite network in
    which that unit is dead, bit for bit.  A row that is not there must not
    activate the first unit by its bias."""
    from paper_2510_17785_gb300 import pmg
    rng = np.random.default_rng(n)
    f32 = dict(dtype=torch.float32, device="cuda")
    theta = mlp.init_params(5).astype(np.float32)
    k, h = 11, 40
    theta[W1 + k * NF:W1 + (k + 1) * NF] = -1.0        # inputs in [1, 2]: unit k is off for every sample
    theta[B1 + k] = 1.0                                # and would be on for a row of zeros
    infinite, finite = theta.copy(), theta.copy()
    infinite[W2 + h * NH + k] = np.inf
    finite[B2 + h] = -1e30
    X = torch.tensor(rng.uniform(1.0, 2.0, (n, NF)), **f32)
    T = torch.tensor(rng.standard_normal((n, 2)), **f32)
    norm = torch.tensor(np.concatenate([np.zeros(NF), np.ones(NF), np.zeros(2), np.ones(2)]), **f32)
    la, ga = pmg.mlp_grad(torch.tensor(infinite, **f32), norm, X, T)
    lb, gb = pmg.mlp_grad(torch.tensor(finite, **f32), norm, X, T)
    assert torch.isfinite(ga).all() and torch.equal(ga, gb) and torch.equal(la, lb)
