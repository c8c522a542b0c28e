"""Training kernels over the ranges of their tile counts: the gradient's sum
over the tiles (chunks of 64), one tile or two per block (from the number of
SMs on, the last block half empty), and the Adam step taken in the sum."""
import numpy as np
import pytest

from oracle import closure_oracle as C
from paper_1211_2205_gb300 import capi
from test_gpu_closure import BF16_TOL, ENGINES, _dev, _oracle_mlp, _params, _rel, bf16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("engine", ENGINES)
@pytest.mark.parametrize("tiles,rest", [(63, 1), (64, 128), (65, 3), (129, 127), (153, 77), (305, 128)])
def test_gradient_and_adam_over_many_tiles(engine, tiles, rest):
    """Against the FP64 oracle with the same BF16 weights and inputs, at the
    bar of the gradient parity (BF16 activations); the Adam step against the
    oracle's optimiser on the same gradient (FP32 arithmetic, 2e-6 at
    lr = 2e-3, the optimiser's bar)."""
    B = (tiles - 1) * 128 + rest
    rng = np.random.default_rng(B)
    X = rng.normal(size=(B + 5, C.N_IN)).astype(np.float32)
    T = rng.normal(size=(B + 5, C.N_OUT)).astype(np.float32)
    idx = rng.permutation(B + 5)[:B].astype(np.int32)
    params = _params(9, scale_out=0.7)
    net = capi.Network(params)
    net.set_engine(engine)
    g = torch.full((capi.MLP_PARAMS,), float("nan"), device="cuda")
    loss = torch.zeros(2, device="cuda")
    Xd, Td, Id = _dev(X), _dev(T), _dev(idx)
    torch.cuda.synchronize()
    net.loss_grad(Xd, Td, B, g, loss, idx=Id)
    net.train_step(Xd, Td, B, 2e-3, loss=loss[1:], idx=Id)
    net.sync()
    got = capi.params_to_dict(g.cpu().numpy())
    ref_loss, ref = C.loss_and_grad(_oracle_mlp(params), bf16(X[idx]).astype(np.float64), T[idx].astype(np.float64))
    l = loss.cpu().numpy()
    assert l[0] == l[1] and abs(l[0] - ref_loss) <= BF16_TOL * ref_loss
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        assert _rel(got[k], ref[k]) <= BF16_TOL, k
    p = capi.params_to_dict(params)
    C.Adam(p, lr=2e-3).step(p, got)
    after = net.params
    np.testing.assert_allclose(after, capi.params_from_dict(p), rtol=0, atol=2e-6)
    # the BF16 weights the kernels use are the new parameters'
    fresh = capi.Network(after)
    fresh.set_engine(engine)
    y = [torch.full((256 * C.N_OUT,), float("nan"), device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    for n, out in zip((net, fresh), y):
        n.forward(Xd, 256, out)
        n.sync()
    assert torch.equal(*y)
