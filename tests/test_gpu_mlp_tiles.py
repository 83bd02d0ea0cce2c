"""The warm-start network where its products go from tiles of 32 columns to
tiles of 128 (152 wide tiles: the output layer at 2,305 or more outputs and
897 or more rows), with rows and columns that fill no tile: predictions and
gradients against the oracle with the same BF16 operands, at the bars of the
smaller networks (2e-3, 5e-3), and nothing written outside the predictions."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2301_04869_gb300 import ipm
    ipm.load()
    return ipm


def nrel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("d_in,d_out,B", [(33, 1, 1), (130, 2304, 1000), (130, 2305, 1000), (97, 2431, 897)])
def test_predictions_and_gradients(gpu, d_in, d_out, B):
    import torch
    dims = (d_in, 128, d_out)
    rng = np.random.default_rng(7)
    m = gpu.MLP(*dims, max_batch=B, seed=0)
    m.set_params((0.05 * rng.normal(0, 1, m.n_params)).astype(np.float32))
    norm = (rng.normal(0, 0.3, d_in), rng.uniform(0.5, 2, d_in), rng.normal(0, 0.3, d_out), rng.uniform(0.5, 2, d_out))
    norm = tuple(v.astype(np.float32) for v in norm)
    m.set_normalization(*norm)
    norm = tuple(v.astype(np.float64) for v in norm)
    p = m.get_params().astype(np.float64)
    X = rng.normal(0, 1, (B, d_in)).astype(np.float32)
    T = rng.normal(0, 1, (B, d_out)).astype(np.float32)
    buf = torch.full((B * d_out + 64,), 3.0, dtype=torch.float32, device="cuda")
    m.forward(torch.from_numpy(X).cuda(), out=buf[32:])
    y = buf.cpu().numpy()
    assert (y[:32] == 3.0).all() and (y[-32:] == 3.0).all()
    yo, _ = omlp.forward(p, X.astype(np.float64), dims, norm, bf16=True)
    assert nrel(y[32:-32].reshape(B, d_out), norm[2] + norm[3] * yo) <= 2e-3
    loss, g = m.gradients(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    Lo, go = omlp.loss_and_grad(p, X.astype(np.float64), T.astype(np.float64), dims, norm, bf16=True)
    assert abs(loss - Lo) <= 1e-4 * Lo
    for a, b in zip(omlp.unflatten(g.astype(np.float64), *dims), omlp.unflatten(go, *dims)):
        assert nrel(a, b) <= 5e-3
