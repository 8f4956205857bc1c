"""The training kernels at the ends of their ranges."""
import numpy as np
import pytest

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("batch", [9, (1 << 32) - 7])
def test_gradient_of_a_batch_as_large_as_its_count(batch):
    """All samples alike, a network of zeros, every target 1: the loss is 1 and
    the only gradient is -2, of the first output's bias.  Terms are powers of
    two, at most 2^24 of them in a 32-bit sum, so what is left are the roundings
    of batch (relative 2^-24, in 1/B) and of eight warps' sums: below 10 * 2^-24."""
    if torch.cuda.mem_get_info()[0] < 41 * batch:
        pytest.skip("not enough free device memory")
    x = torch.zeros(batch, 8, device="cuda")
    target = torch.ones(batch, device="cuda")
    arm = torch.zeros(batch, dtype=torch.int32, device="cuda")
    grad, loss = sp.mlp_backward(torch.zeros(sp.POLICY_WEIGHTS, device="cuda"), x, target, arm)
    grad = grad.cpu().numpy()
    del x, target, arm
    torch.cuda.empty_cache()
    assert abs(float(loss.item()) - 1.0) <= 10 * 2.0 ** -24
    assert abs(grad[-4] + 2.0) <= 20 * 2.0 ** -24
    assert (np.delete(grad, -4 % grad.size) == 0).all()


@pytest.mark.parametrize("batch", [1, 9])
def test_an_odd_sample_is_alone(batch):
    """A first layer that is zero on every sample and overflows the second where
    there is none: all activations are zero, so the only gradient is the first
    output bias's, 2 (0 - 1), exactly up to the roundings of 1/B and the sums."""
    w = torch.zeros(sp.POLICY_WEIGHTS, device="cuda")
    w[0], w[256] = -2e38, 2e38  # W1[0][0], b1[0]
    w[288] = 2.0  # W2[0][0]
    x = torch.zeros(batch, 8, device="cuda")
    x[:, 0] = 1.0
    arm = torch.zeros(batch, dtype=torch.int32, device="cuda")
    grad, loss = sp.mlp_backward(w, x, torch.ones(batch, device="cuda"), arm)
    grad = grad.cpu().numpy()
    assert abs(float(loss.item()) - 1.0) <= 10 * 2.0 ** -24
    assert abs(grad[-4] + 2.0) <= 20 * 2.0 ** -24
    assert (np.delete(grad, -4 % grad.size) == 0).all()


@pytest.mark.parametrize("count", [129, (1 << 32) - 7])
def test_forward_of_a_batch_as_large_as_its_count(count):
    """Outputs of the first and last samples: the output biases, exactly."""
    if torch.cuda.mem_get_info()[0] < 49 * count:
        pytest.skip("not enough free device memory")
    w = torch.zeros(sp.POLICY_WEIGHTS, device="cuda")
    w[-4:] = torch.arange(1.0, 5.0)
    y = sp.mlp_forward(w, torch.zeros(count, 8, device="cuda"))
    ends = torch.cat([y[:3], y[-3:]]).cpu()
    del y
    torch.cuda.empty_cache()
    assert (ends == torch.arange(1.0, 5.0)).all()


@pytest.mark.parametrize("count", [257, (1 << 32) - 7])
def test_adam_of_as_many_weights_as_its_count(count):
    """A first step from zero moments moves every weight by the rate (both bias
    corrections cancel the decay factors, eps is 0), up to the roundings of
    about eight operations."""
    if torch.cuda.mem_get_info()[0] < 17 * count:
        pytest.skip("not enough free device memory")
    w, m1, m2 = (torch.zeros(count, device="cuda") for _ in range(3))
    grad = torch.ones(count, device="cuda")
    sp.mlp_adam(w, grad, m1, m2, lr=0.5, step=1, eps=0.0)
    ends = torch.cat([w[:3], w[-3:]]).cpu()
    del w, m1, m2, grad
    torch.cuda.empty_cache()
    assert ((ends + 0.5).abs() <= 0.5 * 2.0 ** -20).all()
