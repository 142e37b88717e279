"""The Python wrappers without a device: what they accept and what they hand to the library, with a stand-in for the
workspace where one is needed."""
from types import SimpleNamespace

import numpy as np
import pytest

import paper_2412_03378_gb300 as vg


@pytest.mark.parametrize("t", [[1.0, 2.0, 3.0], [1.0, 2.0, 3.0, 1.0], np.array([1.0, 2.0, 3.0, 1.0], np.float32)])
def test_camera_translation_may_be_homogeneous(t):
    """The first three entries of t are read, and the first nine of R."""
    cam = SimpleNamespace(R=np.eye(3), t=t, fx=10.0, fy=11.0, cx=2.0, cy=3.0, width=4, height=5)
    c = vg.camera_struct(cam)
    assert list(c.t) == [1.0, 2.0, 3.0] and list(c.R) == [1, 0, 0, 0, 1, 0, 0, 0, 1]
    cam.R = [[1, 0, 0], [0, 1, 0], [0, 0, 1], [7, 7, 7]]
    assert list(vg.camera_struct(cam).R) == [1, 0, 0, 0, 1, 0, 0, 0, 1]


class StandIn:
    """A workspace that records its calls and writes ones into the outputs, of which the library writes `rows` rows."""

    def __init__(self, rows=None):
        self.generation, self.calls, self.rows = 0, [], rows

    def _fill(self, tensors):
        for t in tensors:
            if t is not None:
                t.view(-1)[:t.numel() if self.rows is None else self.rows * max(1, t[0].numel())] = 1.0

    def project_tomo(self, g, beam, opts, proj, dL=None, *grads, stream=None):
        self.generation += 1
        self.calls.append((opts.flags, dL))
        proj.fill_(0.5)
        self._fill(grads)

    def preprocess(self, g, cams, opts, stream=None):
        self.generation += 1

    def bin_sort(self, stream=None):
        pass

    def render_fwd(self, rgb, T=None, stream=None):
        rgb.fill_(0.25)
        T.fill_(0.5)

    def render_bwd_set(self, dL_drgb, dL_dT, *grads, stream=None):
        self.calls.append((dL_drgb, dL_dT))
        self._fill(grads)

    def query(self):
        raise AssertionError("a query synchronises")


def _params(n=5, sh=4):
    import torch
    return [torch.rand(s) for s in ((n, 3), (n, 3), (n, 4), (n,), (n, sh, 3))]


def _beam():
    return SimpleNamespace(angles=[0.0, 1.0], det_w=6, det_h=4, pitch_u=0.1, pitch_v=0.1, u0=0.0, v0=0.0)


@pytest.fixture
def stand_in(monkeypatch):
    ws = StandIn()
    monkeypatch.setattr(vg, "Workspace", lambda: ws)
    return ws


@pytest.mark.parametrize("how", ["inference", "inference leaf", "no_grad"])
def test_parallel_without_a_gradient(stand_in, how):
    """Computed parameters under inference mode have no version counter; nothing is kept for a backward that cannot come."""
    import torch
    pro, (mu, ls, q, k, _) = vg.Projector(), _params()
    mu.requires_grad_(how == "no_grad")
    with torch.no_grad() if how == "no_grad" else torch.inference_mode():
        if how == "inference leaf":
            mu = torch.rand((5, 3))
        proj = pro.parallel(mu, ls.exp(), torch.nn.functional.normalize(q, dim=1), k, _beam())
    assert proj.shape == (2, 4, 6) and float(proj.min()) == 0.5


def test_gradients_of_what_the_library_does_not_write(monkeypatch):
    """Rows beyond the Gaussians that mu counts, and coefficients beyond sh_degree's, have gradient zero."""
    import torch
    n = 3
    ws = StandIn(rows=n)
    monkeypatch.setattr(vg, "Workspace", lambda: ws)
    empty = torch.empty_like
    monkeypatch.setattr(torch, "empty_like", lambda *a, **k: empty(*a, **k).fill_(float("nan")))
    mu, scale, quat, kappa, _ = _params(n + 2)
    mu = mu[:n].contiguous().requires_grad_(True)
    scale, quat, kappa = (t.requires_grad_(True) for t in (scale, quat, kappa))
    for got in torch.autograd.grad(vg.Projector().parallel(mu, scale, quat, kappa, _beam()).sum(), (mu, scale, quat, kappa)):
        assert torch.equal(got[:n], torch.ones_like(got[:n])) and float(got[n:].abs().sum()) == 0.0
    sh = torch.rand((n, 16, 3), requires_grad=True)
    cams = [SimpleNamespace(width=4, height=3)]
    ws._fill = lambda ts: [t.view(-1)[:t.numel() if t.dim() < 3 else 4 * n * 3].fill_(1.0) for t in ts]
    rgb, _ = vg.Rasterizer().render(mu, scale, quat, kappa, sh, cams, sh_degree=1)
    assert float(torch.autograd.grad(rgb.sum(), sh)[0].sum()) == 4 * n * 3


def test_render_backward_of_T_alone(stand_in):
    """A loss of T alone asks the device nothing (the stand-in's query raises) and hands over a zero dL/drgb."""
    import torch
    params = [p.requires_grad_(True) for p in _params()]
    _, T = vg.Rasterizer().render(*params, [SimpleNamespace(width=4, height=3), SimpleNamespace(width=2, height=1)])
    torch.autograd.grad(T.sum(), params)
    drgb, dT = stand_in.calls[-1]
    assert drgb.shape == (14, 3) and not drgb.any() and torch.equal(dT, torch.ones(14))


@pytest.mark.parametrize("call", ["project_tomo", "tomo_l2_step", "query_density"])
def test_refused_call_leaves_the_outstanding_forward(call):
    """A call that the library refuses for its arguments has not touched the workspace."""
    import ctypes

    ws = vg.Workspace.__new__(vg.Workspace)
    ws.h, ws.generation = None, 7
    refuse = lambda *a: 1
    ws._L = SimpleNamespace(vg_project_tomo=refuse, vg_tomo_l2_step=refuse, vg_query_density=refuse,
                            vg_last_error=lambda h: b"refused")
    g = SimpleNamespace(c=lambda: ctypes.c_int(0))
    args = {"project_tomo": (g, _beam(), vg.Opts(), None), "query_density": (g, (0, 0, 0), (1, 1, 1), (1, 1, 1), vg.Opts(), None),
            "tomo_l2_step": (g, _beam(), vg.Opts(), None, 1.0, None, None, None, None, None, None)}[call]
    stream, vg._stream = vg._stream, lambda s=None: None
    try:
        with pytest.raises(vg.VGError):
            getattr(ws, call)(*args)
    finally:
        vg._stream = stream
    assert ws.generation == 7
