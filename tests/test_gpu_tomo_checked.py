"""Parameters written to between Projector.parallel and its backward in a way that leaves no trace on the tensors (through
.data, or by a kernel outside of torch): the gradient is that of the parameters as they are, as the library's own call
gives it, up to the order of the sums over angles (1e-5 of the largest).  With the angles in one batch and in two."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,angles", [(300, 5), (60000, 71)])
@pytest.mark.parametrize("written", ["nothing", "one mean", "density", "back"])
def test_parameters_written_through_data(gpu_lib, written, n, angles):
    import torch

    vg = gpu_lib
    scene, beam = synth.tomo_scene(n, 251), synth.parallel_beam(angles, det=40, extent=2.0)
    params = [torch.tensor(a, device="cuda:0", requires_grad=True) for a in (scene.mu, scene.scale, scene.quat, scene.kappa)]
    pro = vg.Projector()
    dL = torch.rand((angles, 40, 40), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(6))
    total = (pro.parallel(*params, beam) * dL).sum()
    first = pro.ws.read_bins()
    if written == "one mean":
        params[0].data[n // 2] *= 0.5
    elif written == "density":
        params[3].data.mul_(3.0)
    elif written == "back":
        params[3].data.mul_(2.0).mul_(0.5)
    got = [torch.autograd.grad(total, params, retain_graph=True) for _ in range(2)]
    ws, proj = vg.Workspace(), torch.empty((angles, 40, 40), device="cuda:0")
    want = [torch.zeros(p.shape, device="cuda:0") for p in params]
    ws.project_tomo(vg.Gaussians(*(p.detach() for p in params), None, 0), beam, vg.Opts(tau_cut=1e-6), proj, dL, *want)
    for g in got:
        for x, y in zip(g, want):
            assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())
    for a, b in zip(pro.ws.read_bins(), ws.read_bins()):
        assert (a == b).all()
    if written in ("nothing", "back"):
        for a, b in zip(first, ws.read_bins()):
            assert (a == b).all()
