"""Calls that follow one another in a stream without the host in between.  Every kernel of a layer is launched ahead of its
predecessor's end, so the combine is on the GPU while the dispatch still writes the handle that it reads."""
import pytest
import torch

import harness as Hn
from paper_2607_06202_b200 import binding as B
from paper_2607_06202_b200 import workload as W

pytestmark = pytest.mark.gpu


class Layers:
    """Layers of different routing, one after the other on one buffer, with what each returns when the host waits in between."""

    def __init__(self, T, H, E, R, k, payload=0, dedup=0, layers=4):
        self.wls = [W.make_workload(W.Config("chain", T=T, H=H, E=E, R=R, k=k, payload=payload, dedup=dedup, seed=100 + i))
                    for i in range(layers)]
        cfg = self.wls[0].cfg
        refs = [Hn.oracle_reference(wl, num_threads=8) for wl in self.wls]
        self.cap = max(cap for _, _, cap, _ in refs)
        self.buf = Hn.make_buffer(cfg, self.cap)
        self.dev = [Hn.device_inputs(wl)[:3] for wl in self.wls]
        gen = torch.Generator(device="cuda").manual_seed(7)
        self.ys = [torch.randn((R, self.cap, H), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(layers)]
        self.outs = [torch.empty((T, H), dtype=torch.bfloat16, device="cuda") for _ in range(layers)]
        self.want = []
        for (x, idx, w), y in zip(self.dev, self.ys):
            self.buf.dispatch(x, idx, w)
            torch.cuda.synchronize()
            self.want.append(self.buf.combine(y, w).clone())
            torch.cuda.synchronize()
        # the first of them against the oracle: the others are told apart by it
        import oracle
        (ids, lay, _, _), wl = refs[0], self.wls[0]
        bits = self.ys[0].view(torch.int16).cpu().numpy().view("uint16")
        Hn.check_combine(self.want[0], oracle.combine(bits, ids, wl.topk_w, lay.slot_row, E, R, num_threads=8)[0])
        assert not torch.equal(self.want[0], self.want[1])

    def run(self):
        for (x, idx, w), y, out in zip(self.dev, self.ys, self.outs):
            self.buf.dispatch(x, idx, w)
            self.buf.combine(y, w, out=out)

    def check(self):
        torch.cuda.synchronize()
        assert self.buf.status() == 0
        for i, (out, want) in enumerate(zip(self.outs, self.want)):
            assert torch.equal(out.view(torch.int16), want.view(torch.int16)), f"layer {i}"
            out.zero_()


SHAPES = [(1200, 1024, 64, 8, 8, 0, 0), (2000, 512, 64, 16, 6, 0, 1), (1100, 1024, 32, 4, 8, 1, 1), (8300, 256, 16, 4, 1, 0, 0),
          (2100, 512, 40, 8, 5, 0, 1), (6000, 2048, 64, 8, 8, 0, 0), (4200, 4096, 128, 16, 8, 1, 0), (128, 512, 32, 8, 4, 0, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_layers_of_different_routing(shape):
    """Large calls (both ways the combine reads rows, every instance of the number of slots) and a small one."""
    s = Layers(*shape)
    for _ in range(3):
        s.run()
        s.check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.run()
    for _ in range(5):
        graph.replay()
    s.check()


@pytest.mark.parametrize("T", [200, 3000])
def test_captured_behind_other_kinds_of_work(T):
    """A combine behind work that another stream joins in, a copy and a fill; a dispatch behind the same."""
    s = Layers(T, 512, 32, 8, 4, layers=2)
    idx, y = s.dev[0][1].clone(), s.ys[0].clone()
    side = torch.cuda.Stream()

    def layer(i, how):
        x, idx_i, w = s.dev[i]
        main = torch.cuda.current_stream()
        if how == "join":
            side.wait_stream(main)
            with torch.cuda.stream(side):
                idx.copy_(idx_i)
            scratch.add_(1)
            main.wait_stream(side)
        else:
            idx.copy_(idx_i)
        s.buf.dispatch(x, idx, w)
        if how == "join":
            side.wait_stream(main)
            with torch.cuda.stream(side):
                torch.add(s.ys[i], 0, out=y)
            scratch.add_(1)
            main.wait_stream(side)
        else:
            y.copy_(s.ys[i])
            s.outs[i].zero_()
        s.buf.combine(y, w, out=s.outs[i])

    scratch = torch.zeros(64, device="cuda")
    for how in ("join", "copies"):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            layer(0, how)
            layer(1, how)
        for _ in range(3):
            graph.replay()
        s.check()
