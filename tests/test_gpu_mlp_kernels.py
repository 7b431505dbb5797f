"""The proposal network's gradient and inference kernels at the edges of their tiles (32 rows; the gradient's blocks
take several tiles from 304 tiles on, 9,728 rows), with buffers that are not aligned for wide accesses."""
import numpy as np
import pytest

from oracle import mlp
from paper_1811_03510_gb300 import ccs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_03510_gb300 import build_ext
    build_ext.build()
    torch.cuda.set_device(0)


def shifted(shape, dtype, k):
    """An uninitialised tensor that starts k elements after an aligned address."""
    n = int(np.prod(shape))
    return torch.empty(n + k, dtype=dtype, device="cuda")[k:].view(shape)


# (1e-4 and 1e-5 are the bounds that the gradient has against the FP64 oracle elsewhere: sums of up to 12,000 FP32 terms)
@pytest.mark.parametrize("B", [1, 31, 32, 33, 700, 9728, 12001])
def test_gradient_at_the_edges_of_its_tiles(B):
    rng = np.random.default_rng(B)
    p = ccs.ccs_proposal_create(seed=4)
    theta = ccs.ccs_proposal_get_params(p).astype(np.float64)
    X, y = rng.normal(size=(B, 24)).astype(np.float32), rng.integers(0, 64, size=B).astype(np.uint8)
    dX, dy = shifted((B, 24), torch.float32, 1), shifted((B,), torch.uint8, 3)
    dX.copy_(torch.from_numpy(X))
    dy.copy_(torch.from_numpy(y))
    grad, loss = shifted((9920,), torch.float32, 1), torch.zeros(1, device="cuda")
    ccs.ccs_proposal_grad(p, dX, dy, B, grad, loss)
    torch.cuda.synchronize()
    L_ref, g_ref = mlp.loss_and_grad(theta, X.astype(np.float64), y)
    assert abs(loss.item() - L_ref) <= 1e-5 * abs(L_ref)
    g = grad.cpu().numpy().astype(np.float64)
    for part, ref in zip(mlp.unpack(g), mlp.unpack(g_ref)):
        assert np.linalg.norm(part - ref) <= 1e-4 * max(np.linalg.norm(ref), 1e-30)
    # the same gradient every time (no atomics), and a training step publishes what it trained
    again = torch.empty_like(grad)
    ccs.ccs_proposal_grad(p, dX, dy, B, again)
    torch.cuda.synchronize()
    assert torch.equal(grad, again)
    ccs.ccs_proposal_train_step(p, dX, dy, B, 1e-3)
    q = ccs.ccs_proposal_create(seed=9)
    ccs.ccs_proposal_set_params(q, ccs.ccs_proposal_get_params(p))
    out = [torch.empty(B, 64, device="cuda") for _ in range(2)]
    for h, o in zip((p, q), out):
        ccs.ccs_proposal_infer(h, dX, B, o)
    torch.cuda.synchronize()
    assert torch.equal(*out)
    for h in (p, q):
        ccs.ccs_proposal_destroy(h)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 129, 58400])
def test_inference_rows_do_not_depend_on_their_tile(n):
    p = ccs.ccs_proposal_create(seed=5)
    m = 1 << 16
    X = torch.randn(m, 24, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
    ref = [torch.empty(m, 64, device="cuda"), torch.empty(m, dtype=torch.uint8, device="cuda"), torch.empty(m, device="cuda")]
    ccs.ccs_proposal_infer(p, X, m, *ref)
    a = 7   # rows 7 .. 7 + n, in buffers that start at odd multiples of their element
    Y = shifted((n, 24), torch.float32, 1)
    Y.copy_(X[a:a + n])
    out = [shifted((n, 64), torch.float32, 1), shifted((n,), torch.uint8, 1), shifted((n,), torch.float32, 1)]
    ccs.ccs_proposal_infer(p, Y, n, *out)
    torch.cuda.synchronize()
    for got, want in zip(out, ref):
        assert torch.equal(got, want[a:a + n])
    # each result alone
    for k in range(3):
        one = [None, None, None]
        one[k] = torch.empty_like(out[k])
        ccs.ccs_proposal_infer(p, Y, n, *one)
        torch.cuda.synchronize()
        assert torch.equal(one[k], out[k])
    ccs.ccs_proposal_destroy(p)
