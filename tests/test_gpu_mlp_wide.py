"""Forward pass of the atom-pair MLP with an output layer wider than one grid's
columns (65535 tiles of 64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_forward_of_a_wide_layer():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    from oracle import mlp_ref
    nout, rows = 65535 * 64 + 70, 2
    net = fk.MLP(1, 2, nout, rows, seed=5)
    p = net.params().astype(np.float64)
    p[-nout:] = np.linspace(-1.0, 1.0, nout)
    net.set_params(p.astype(np.float32))
    X = np.array([[0.3], [-1.2]], dtype=np.float32)
    Y = net.forward(torch.tensor(X, device="cuda")).cpu().numpy()
    net.close()
    ref = mlp_ref.forward(p.astype(np.float32).astype(np.float64), X.astype(np.float64), 1, 2, nout, weights_bf16=True)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.abs(Y - ref).max() <= 1e-5 * np.abs(ref).max()
