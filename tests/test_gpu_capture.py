"""Steps captured into a CUDA graph by the caller: consecutive steps (joined by a
programmatic edge), steps after a memset, a copy and a torch kernel, and a step that
joins two streams; every replay gives the bits of the same calls made directly."""
import numpy as np
import pytest
import torch

from paper_2009_04619_gb300 import seisgb
from gpu_util import ensure_lib, to_padded

pytestmark = pytest.mark.gpu

STORAGE = {"fp32": (seisgb.FP32, torch.float32), "fp16": (seisgb.FP16_SCALED, torch.float16),
           "bf16": (seisgb.BF16, torch.bfloat16), "fp32_diff": (seisgb.FP32_DIFF, torch.float32),
           "bf16_diff": (seisgb.BF16_DIFF, torch.bfloat16)}


class _Fields:
    """Random fields of one grid and the step that advances them: n reads f[n & 1]."""

    def __init__(self, fmt, ext=(72, 40, 30, 6), seed=0):
        ensure_lib()
        storage, t = STORAGE[fmt]
        nx, ny, nz, nb = ext
        g32 = seisgb.make_grid(nx, ny, nz, nb, 10.0, 10.0, 10.0, 5e-4, 3000.0)
        self.g = seisgb.make_grid(nx, ny, nz, nb, 10.0, 10.0, 10.0, 5e-4, 3000.0, 1e-3, storage)
        rng = np.random.default_rng(seed)
        pad = lambda a: to_padded(g32, a.astype(np.float32))
        a, b = (pad(rng.standard_normal(g32.shape)) for _ in range(2))
        top = [float(x.abs().max()) for x in (a, b)]
        self.diff = fmt.endswith("diff")
        self.f = [a.to(t), b.to(t)]
        self.d = (0.1 * b).to(t)
        self.m = pad((rng.uniform(1500, 3000, g32.shape) * 5e-4) ** 2)
        self.phi = pad(np.zeros(g32.shape))
        # scales of one: the values stay far below the largest fp16
        self.scale = torch.tensor([1.0] * 4 + [top[0], 0.0, 0.0, top[1]], device="cuda")
        self.has_scale = fmt == "fp16"
        self.src = (nb + 3, nb + 2, nb + 1, torch.full((64,), 50.0, device="cuda"))
        torch.cuda.synchronize()

    def state(self):
        return [*self.f, self.d, self.phi, self.scale]

    def step(self, n):
        u, v = self.f[n & 1], self.f[(n + 1) & 1]
        if self.diff:
            seisgb.stencil_step_diff(self.g, u, v, self.d, self.m, self.phi, n, self.src)
        else:
            seisgb.stencil_step(self.g, u, v, self.m, self.phi, n, self.src,
                                scale_state=self.scale if self.has_scale else None)


def _captured_equals_direct(make, work, replays=2):
    """work(fields) run `replays` times directly, and captured once and replayed."""
    direct = make()
    for _ in range(replays):
        work(direct)
    torch.cuda.synchronize()
    fields = make()
    graph = torch.cuda.CUDAGraph()
    before = [x.clone() for x in fields.state()]
    with torch.cuda.graph(graph):
        work(fields)
    for x, y in zip(fields.state(), before):  # capturing runs nothing
        assert torch.equal(x, y)
    for _ in range(replays):
        graph.replay()
    torch.cuda.synchronize()
    seisgb.device_status()
    for x, y in zip(fields.state(), direct.state()):
        assert torch.equal(x, y)
    assert not torch.equal(fields.state()[0], before[0])


@pytest.mark.parametrize("fmt", list(STORAGE))
def test_consecutive_steps(fmt):
    def work(s):
        for n in range(4):  # a multiple of four: the scale state's slots repeat
            s.step(n)
    _captured_equals_direct(lambda: _Fields(fmt), work)


@pytest.mark.parametrize("fmt", ["fp32", "bf16"])
def test_steps_between_memset_copy_and_kernel_nodes(fmt):
    def work(s):
        s.phi.zero_()
        s.step(0)
        keep = s.f[1].clone()
        s.step(1)
        s.f[0].copy_(keep)  # a copy node right before a step
        s.step(2)
        s.f[1].mul_(0.5)  # a kernel that triggers no dependents
        s.step(3)
    _captured_equals_direct(lambda: _Fields(fmt), work)


def test_step_after_a_cross_stream_join():
    """Two shots' steps on two streams; a third shot's step waits for both and reads a
    sum of their fields."""
    class Three:
        def __init__(self):
            self.s = [_Fields("fp32", seed=q) for q in range(3)]
            self.side = torch.cuda.Stream()

        def state(self):
            return [x for s in self.s[::-1] for x in s.state()]

    def work(t):
        a, b, c = t.s
        main = torch.cuda.current_stream()
        t.side.wait_stream(main)
        for n in range(2):
            a.step(n)
        with torch.cuda.stream(t.side):
            for n in range(2):
                b.step(n)
        main.wait_stream(t.side)
        c.step(0)  # joins both streams' last steps
        torch.add(a.f[0], b.f[0], alpha=0.5, out=c.f[0])
        c.step(1)
    _captured_equals_direct(Three, work)
