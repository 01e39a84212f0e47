"""Parameters and results in tensors that are not on the problem's device (here: in host memory) go through a
copy: the same bits as with the problem's own device, whose tensors the kernels read and write themselves."""
import pytest
import torch

import scenegen
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("params, loss_on, grad_on", [("cpu", "cuda", "cuda"), ("cuda", "cpu", "cuda"),
                                                      ("cuda", "cuda", "cpu"), ("cpu", "cpu", "cpu")])
def test_host_tensors(params, loss_on, grad_on):
    build.build()
    sc = scenegen.make_scene("ring16", seed=4)
    R, t = sc.R_init, sc.t_init
    C = -(R.transpose(1, 2) @ t[:, :, None])[:, :, 0] + 0.01
    with fm.Problem(sc.R_init, sc.t_init, sc.cam_i, sc.cam_j, sc.pair_id, sc.x1, sc.x2) as p:
        p.set_params_device(R.cuda(), C.cuda())
        loss, grad = p.loss_grad()
        p.set_params_device(R.cuda(), (C + 0.1).cuda())
        p.set_params_device(R.to(params), C.to(params))
        lo = torch.zeros(1, dtype=torch.float64, device=loss_on)
        go = torch.zeros(sc.n_cams, 6, dtype=torch.float64, device=grad_on)
        p.loss_grad_device(lo, go)
        assert lo.item() == loss and torch.equal(go.cpu(), torch.from_numpy(grad))
        go.zero_()
        p.loss_grad_device(None, go)
        assert torch.equal(go.cpu(), torch.from_numpy(grad))
