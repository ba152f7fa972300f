"""The indicator's network kernels at the edges of their 64-sample tiles and of
their persistent grid, from aligned and unaligned feature arrays, and the
training data of uniform sub-grids, against the CPU oracle.

Tolerances: a gradient entry is a chain of at most a few hundred FP32
additions per CTA and of 456 partials, so 1e-4 of the largest entry holds it
with two decimal digits to spare; an output of the forward pass changes by
less than 1e-5 with the order of its sums, and where the first hidden layer
rounds to the other BF16 neighbour by at most 2^-8 |h w| per unit, which the
weights here keep under 1e-3."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
GAMMA = 5.0 / 3.0


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2107_10987_gb300 import _build, hydro
    _build.build()
    return hydro


# one sample, a tile's edges, the partials' edges, more tiles than CTAs
@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 128, 129, 456 * 64 + 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward_and_gradient_at_tile_edges(H, oracle_mod, n, shift):
    from oracle import gate
    rng = np.random.default_rng(n)
    theta = rng.normal(0, 0.1, gate.NPARAM).astype(np.float32)
    X = rng.uniform(-1, 1, (n, 54)).astype(np.float32)
    y = (rng.uniform(size=n) < 0.3).astype(np.float32)
    buf = torch.zeros(n * 54 + 1, dtype=torch.float32, device="cuda")
    Xt = buf[shift:shift + n * 54].view(n, 54)  # shift 1: not even 8-byte aligned
    Xt.copy_(torch.tensor(X))
    p, yt = torch.tensor(theta, device="cuda"), torch.tensor(y, device="cuda")
    grad, loss = torch.empty_like(p), torch.empty(1, dtype=torch.float32, device="cuda")
    out = torch.full((n + 1,), -7.0, dtype=torch.float32, device="cuda")
    H.hydro_mlp_loss_grad(p, Xt, yt, grad, loss, 4.0, 0.5)
    H.hydro_mlp_forward(p, Xt, out[:n])
    again = torch.empty_like(grad)
    H.hydro_mlp_loss_grad(p, Xt, yt, again, None, 4.0, 0.5)
    torch.cuda.synchronize()
    th = gate.bf16_round(theta)
    Lo, go = gate.loss_and_grad(th, X.astype(np.float64), y.astype(np.float64), 4.0, 0.5)
    assert loss.item() == pytest.approx(Lo, rel=1e-5)
    assert np.max(np.abs(grad.cpu().numpy() - go)) <= 1e-4 * np.max(np.abs(go))
    assert torch.equal(grad, again)  # a fixed order of sums
    oo = gate.forward_infer(th, X.astype(np.float64))
    assert np.max(np.abs(out[:n].cpu().numpy() - oo)) < 1e-3
    assert out[n].item() == -7.0


def test_training_data_of_uniform_subgrids(H, oracle_mod):
    """Uniform padded blocks take a short cut; one changed corner cell, or one
    changed velocity, takes the general path.  All against the oracle."""
    from oracle import gate
    U = np.empty((5, 10, 14, 14, 14))
    for i, (rho, vx, p) in enumerate([(1.0, 0.0, 1e-5), (1.0, 0.0, 1e-5), (1e-10, 0.3, 1e-8), (2.0, -0.5, 3.0),
                                      (1.0, 0.0, 1.0)]):
        full = np.full((14, 14, 14), rho)
        v = np.zeros((3, 14, 14, 14))
        v[0] = vx
        q = np.full((14, 14, 14), p)
        if i == 1:
            full[0, 0, 0] = 1.5
        if i == 3:
            v[1, 7, 7, 7] = 0.25
        if i == 4:
            q[5:8, 5:8, 5] = 2.0
        U[i] = W.conserved_from_primitive(full, v, q, GAMMA)
    Ut = torch.tensor(U, device="cuda")
    B = H.make_batch(Ut, torch.zeros((5, 3), dtype=torch.float64, device="cuda"),
                     torch.full((5,), 0.05, dtype=torch.float64, device="cuda"))
    X = torch.full((5 * 512, 54), 9.0, dtype=torch.float32, device="cuda")
    y = torch.full((5 * 512,), 9, dtype=torch.uint8, device="cuda")
    H.hydro_gate_data(H.Context(GAMMA, 0.0), B, X, y)
    torch.cuda.synchronize()
    U32 = U.astype(np.float32).astype(np.float64)
    assert np.max(np.abs(X.cpu().numpy() - gate.features(U32, GAMMA))) < 2e-6
    assert np.array_equal(y.cpu().numpy(), gate.labels(U32, GAMMA))
    assert y[3 * 512:].any() and not y[:512].any()
