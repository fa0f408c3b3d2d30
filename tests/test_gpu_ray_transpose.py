"""The adjoint of the ray transform uses the forward's own float32 weights: the matrices
of the two, taken column by column from unit images and unit sinograms, are transposes of
each other bit for bit.  Both adjoint kernels are reached (the one that stages tiles needs
two CTAs per SM, so a batch of a few thousand); bins narrower and wider than a pixel."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,A,D", [(16, 6, 23), (9, 7, 61), (12, 30, 40), (20, 5, 9), (33, 4, 47), (2, 8, 3)])
def test_exact_transpose(n, A, D):
    from paper_2006_04591_gb300.ray import RayTransform
    op = RayTransform(n, A, D, device=0)
    eye = lambda k, shape: torch.eye(k, device="cuda").reshape((k,) + shape)  # noqa: E731
    fwd = op.forward(eye(n * n, (n, n))).reshape(n * n, A * D)
    y = eye(A * D, (A, D))
    adj = op.adjoint(y).reshape(A * D, n * n)
    assert torch.equal(fwd.T, adj)
    many = 4096 // (A * D) + 1
    assert torch.equal(op.adjoint(y.repeat(many, 1, 1)).reshape(many, A * D, n * n)[-1], adj)
    one = torch.stack([op.adjoint(y[d:d + 1])[0].reshape(-1) for d in range(0, A * D, 7)])
    assert torch.equal(one, adj[::7])
