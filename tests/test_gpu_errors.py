"""GPU tests of host-side errors: a call that the runtime refuses reports it once, and calls after it run."""
import pytest

from paper_2202_06516_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_refused_launch_does_not_reach_the_next_call():
    """32 images of 512 x 512 need 65,536 tiles along one grid dimension (65,535 are allowed): the
    prediction is refused. A network and a lattice made afterwards start and run."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2202_06516_gb300 import lbm
    x = torch.zeros(32, 512, 512, 8, dtype=torch.bfloat16, device="cuda")
    phi = torch.empty(32, 512, 512, dtype=torch.float32, device="cuda")
    big = lbm.Surrogate(512, 512, base=8, max_batch=32)
    big.set_weights(W.unet_init(8, 0))
    for _ in range(2):
        with pytest.raises(lbm.LbmError, match="invalid"):
            big.forward(x.data_ptr(), 32, phi.data_ptr())
    small = lbm.Surrogate(64, 64, base=8, max_batch=1)
    small.set_weights(W.unet_init(8, 0))
    small.forward(x.data_ptr(), 1, phi.data_ptr())
    with pytest.raises(lbm.LbmError, match="invalid"):
        big.forward(x.data_ptr(), 32, phi.data_ptr())
    lat = lbm.Lattice(64, 64, **W.MODEL)
    lat.set_geometry(drop=(32.0, 20.0, 10.0, 5.6))
    lat.step(4)
    lat.mass()
    big.forward(x.data_ptr(), 31, phi.data_ptr())
    for o in (big, small, lat):
        o.close()
