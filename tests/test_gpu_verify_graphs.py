"""When hydra_verify captures its forward pass, and what keeps the graph.  A replayed call launches one kernel more than a launched one (the copy of
the tokens), which tells them apart."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg

pytestmark = pytest.mark.gpu

CAPTURED_AT = 8


class Driver:
    """A context on a stream of its own; verify(batch) says whether the call was replayed and that its results are those of launched kernels."""

    def __init__(self, max_batch=10):
        from paper_2402_05109_b200 import Hydra
        self.m, self.max_batch = ModelCfg(1, 256, 2, 128, 512, 1024, dtype="bf16"), max_batch
        h = HeadCfg(3, 1, False)
        self.g = Hydra(self.m, h, load_tree("tree15_d3"), {k: v.cuda() for k, v in make_weights(self.m, h, 93).items()}, max_batch, 128)
        self.prompts = [p.cuda() for p in make_prompts(93, [9 + i for i in range(max_batch)], self.m.vocab)]
        self.gen = torch.Generator().manual_seed(7)
        self.stream = torch.cuda.Stream()
        self.batch = 0

    def launches(self, cand):
        before = self.g.launch_count()
        res = self.g.verify(cand, want_logits=True)
        return res, self.g.launch_count() - before

    def verify(self, batch, times=1):
        """Whether each call was replayed."""
        with torch.cuda.stream(self.stream):
            if batch != self.batch:
                self.g.prefill(self.prompts[:batch])
                self.batch = batch
            got = []
            for _ in range(times):
                cand = torch.randint(0, self.m.vocab, (batch, 16), dtype=torch.int32, generator=self.gen).cuda()
                self.g.set_step_graph(False)
                want, plain = self.launches(cand)
                self.g.set_step_graph(True)
                res, n = self.launches(cand)
                assert torch.equal(res[0], want[0]) and torch.equal(res[1], want[1])
                got.append({plain: False, plain + 1: True}[n])
        return got


def test_capture_at_the_eighth_call_of_a_batch():
    d = Driver()
    assert d.verify(1, CAPTURED_AT + 2) == [False] * (CAPTURED_AT - 1) + [True] * 3
    assert d.verify(3, CAPTURED_AT) == [False] * (CAPTURED_AT - 1) + [True]      # a batch of its own, counted from its own first call
    assert d.verify(1, 2) == [True] * 2
    d.g.close()


def test_the_batch_that_was_asked_for_longest_ago_goes():
    d = Driver()
    assert d.verify(1, CAPTURED_AT)[-1]
    for b in range(2, 11):                         # nine others pass by while batch 1 is in use
        assert d.verify(b) == [False] and d.verify(1) == [True]
    for b in range(2, 10):                         # eight others while it is not
        d.verify(b)
    assert d.verify(1) == [False]
    d.g.close()


def test_steps_leave_the_verifications_graphs():
    d = Driver(1)
    assert d.verify(1, CAPTURED_AT)[-1]
    plants = [torch.full((1, 16), -1, dtype=torch.int32, device="cuda") for _ in range(11)]
    with torch.cuda.stream(d.stream):
        d.g.prefill(d.prompts[:1])
        for p in plants:                           # a step graph for each but the first
            d.g.set_plant(p)
            d.g.step()
        d.g.set_plant(None)
    assert d.verify(1) == [True]
    d.g.close()


def test_the_criterion_leaves_the_verifications_graphs():
    """A sampling loop sets the criterion before every verification; the graph ends before the criterion comes in."""
    d = Driver(2)
    assert d.verify(2, CAPTURED_AT)[-1]
    u = torch.tensor([0.25, 0.75], device="cuda")
    for mode, tau in ((1, 0.7), (1, 1.3), (0, 1.0)):
        d.batch = 0                                # a prompt pass: the criterion may then change
        with torch.cuda.stream(d.stream):
            d.g.prefill(d.prompts[:2])
            d.batch = 2
            d.g.set_acceptance(mode, tau, 0.1, 0.3, u if mode else None)
        assert d.verify(2, 2) == [True] * 2
    d.g.set_gemm_mode(1)                           # another kernel: nothing captured survives
    d.g.set_gemm_mode(0)
    assert d.verify(2) == [False]
    d.g.close()
