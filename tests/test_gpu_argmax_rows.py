"""Argmax over many rows of a wide vocabulary (each CTA runs over several spans of a row): the lowest token of the row's largest logit, at row
counts on both sides of the choice and vocabularies that end inside a span."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("vocab", [20608, 32000, 2048 * 9])
def test_lowest_token_of_the_largest_logit(batch, vocab):
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(1, 256, 2, 128, 512, vocab, dtype="bf16")
    h = HeadCfg(4, 1, False)
    w = {k: v.cuda() for k, v in make_weights(m, h, 95, device="cuda").items()}
    w["lm_head"][vocab // 2:] = w["lm_head"][:vocab - vocab // 2].clone()      # every logit twice: ties across spans
    g = Hydra(m, h, load_tree("tree63_d4"), w, batch, 256)
    g.prefill([p.cuda() for p in make_prompts(95, [40 + i for i in range(batch)], vocab)])
    cand = torch.randint(0, vocab, (batch, 64), dtype=torch.int32, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    amax, logits = g.verify(cand, want_logits=True)
    g.poll_status()
    best = logits.max(dim=-1, keepdim=True).values
    first = (logits == best).int().argmax(dim=-1)                               # the first of equal maxima
    assert torch.equal(amax.long(), first.long())
    # the logits themselves: the operand planes hold 16 bits (2^-17 a term), float sums of 256 terms
    ref = g.get_buffer("H_TREE").view(-1, 256)[:batch * 64].double() @ w["lm_head"].double().T
    assert float((logits.view(batch * 64, vocab).double() - ref).abs().max()) <= 2e-4 * float(ref.abs().max())
    assert torch.equal(g.verify(cand), amax)                                    # and without storing the logits
    g.close()
