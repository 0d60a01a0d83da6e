"""Networks of many layers: what they take of the device's memory."""
import pytest

from paper_2411_05799_gb300 import npx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_partial_sums_do_not_grow_with_the_depth():
    """Weights, moments, gradients and the two BF16 copies are 20 bytes a weight, the five arrays of
    activations and their gradients 10 bytes a row and column; the partial sums of the weight gradients
    are those of eight layers (16 FP32 values a weight of a 512 x 512 layer), however many there are."""
    H, layers, M = 512, 40, 128
    torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = npx.MLP(128, 128, n_hidden=H, n_hidden_layers=layers, max_batch=M)
    used = before - torch.cuda.mem_get_info()[0]
    known = 20 * (layers - 1) * H * H + 10 * M * H * layers + 8 * 16 * 4 * H * H
    assert used < 1.1 * known + (64 << 20), (used, known)
    net.close()
