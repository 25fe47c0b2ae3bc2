"""Device memory of a network: gradient buffers are shared by the layers in turn, and what no layer of the
network stores or gathers through a buffer is not allocated."""
import pytest

pytestmark = pytest.mark.gpu


# MiB with one FP32 gradient per activation, one BF16 pre-activation gradient for all layers and an im2col
# buffer in every network: the layers' own BF16 gradients must not take more
@pytest.mark.parametrize("H,Wd,base,B,bound", [(256, 256, 32, 8, 1826), (128, 384, 32, 8, 1452),
                                               (264, 264, 32, 32, 6836)])
def test_network_memory(H, Wd, base, B, bound):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2202_06516_gb300 import lbm
    torch.zeros(1, device="cuda")
    lbm.Surrogate(64, 64, base=8, max_batch=1).close()  # the library's own context and code
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = lbm.Surrogate(H, Wd, base=base, max_batch=B)
    used = (before - torch.cuda.mem_get_info()[0]) / 2**20
    s.close()
    assert used <= bound, used
