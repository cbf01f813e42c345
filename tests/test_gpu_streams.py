"""Calls behind an event of another stream: every kernel of a call's chain sees what the other
stream wrote before the event, and the other stream's next writes wait for the whole call."""
import pytest
import torch

import synth
from tests.helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsct():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_01844_gb300 as g
    from paper_2604_01844_gb300 import build

    build.build()
    return g


def _project(gsct, W, H, tile):
    views = synth.cone_views(6, W, H)
    proj = gsct.Projector(views, W, H, tile=tile)

    def call(mr, sc, qt):
        img = proj.forward(mr, sc, qt)
        return [img], list(proj.backward(mr, sc, qt, torch.ones_like(img)))

    return call


def _voxelize(gsct):
    vox = gsct.Voxelizer(synth.cube_grid(96))

    def call(mr, sc, qt):
        vol = vox.forward(mr, sc, qt)
        return [vol], list(vox.backward(mr, sc, qt, torch.ones_like(vol)))

    return call


def _mlp(gsct):
    from paper_2604_01844_gb300.mlp import BrickMLP

    t = 0.3 * torch.rand(256, 4096, device="cuda", generator=torch.Generator("cuda").manual_seed(2))

    def call(x, _, __):
        net, loss = BrickMLP(seed=4), torch.zeros(1, device="cuda")
        net.train_step(x[:256].to(torch.bfloat16), t, loss, lr=1e-3)
        return [net.flat_grad, net.flat], [loss]

    return call


# both list routes of the rasterizer, the voxelizer's sort, the MLP's GEMM chain
@pytest.mark.parametrize("kind", ["direct", "sorted", "voxelize", "mlp"])
def test_chain_behind_an_event_of_another_stream(gsct, kind):
    """The parameters arrive on a side stream after some 10 ms; the call waits for them by an event
    alone, and the side stream overwrites them behind an event of the call.  Outputs with a fixed
    order of sums equal the undisturbed call's bit for bit; those that meet in atomics within 1e-5 of
    their largest terms (for a rotation the scale gradient times the scale, whose differences make
    it), as undisturbed calls differ among themselves.  Parameters come in at half their size
    before the event, so a missed wait shows in every output."""
    call = {"direct": lambda: _project(gsct, 160, 144, 16), "mlp": lambda: _mlp(gsct),
            "sorted": lambda: _project(gsct, 512, 512, 8), "voxelize": lambda: _voxelize(gsct)}[kind]()
    if kind == "mlp":
        good = [torch.rand(256, 4096, device="cuda", generator=torch.Generator("cuda").manual_seed(1))]
        good += [torch.zeros(1, device="cuda")] * 2
    else:
        good = to_dev(*synth.gaussians(3, 4000))
    other = [0.5 * t for t in good]
    want = call(*good)  # plans the workspaces
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(3):
        buf = [t.clone() for t in other]
        ready, done = torch.cuda.Event(), torch.cuda.Event()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)
            for b, t in zip(buf, good):
                b.copy_(t)
            ready.record(side)
        torch.cuda.current_stream().wait_event(ready)
        got = call(*buf)
        done.record()
        side.wait_event(done)
        with torch.cuda.stream(side):
            for b, t in zip(buf, other):
                b.copy_(t)
        torch.cuda.synchronize()
        for a, b in zip(got[0], want[0]):
            assert torch.equal(a, b)
        for a, b in zip(got[1], want[1]):
            terms = float(b.abs().max())
            if kind != "mlp":
                terms = max(terms, float((want[1][1] * good[1]).abs().max()))
            assert torch.allclose(a, b, rtol=1e-4, atol=1e-5 * terms)
