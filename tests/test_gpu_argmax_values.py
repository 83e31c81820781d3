"""Argmax over many rows, where each CTA runs over several spans and where it does not: vocabularies that are and are not a multiple of four, ties,
infinities of either sign, and logits that are not numbers (which never win)."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 9])
@pytest.mark.parametrize("vocab", [1022, 20609, 20610, 20612])
@pytest.mark.parametrize("special", ["none", "some", "all infinite"])
def test_lowest_token_of_the_largest_logit(batch, vocab, special):
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(1, 256, 2, 128, 512, vocab, dtype="fp32")
    h = HeadCfg(3, 1, False)
    w = make_weights(m, h, 98, device="cuda")
    lm = w["lm_head"]
    lm[vocab // 2:] = lm[:vocab - vocab // 2].clone()        # every logit twice
    one = torch.zeros(256, device="cuda")
    one[3] = float("inf")                                     # a logit of +inf or -inf, by the sign of the hidden row's element
    if special == "some":
        lm[[vocab - 1, vocab // 3, 7]] = one
        lm[[0, 5, vocab - 2, vocab // 3 + 1]] = float("nan")
    if special == "all infinite":
        lm[:] = one
    g = Hydra(m, h, load_tree("tree15_d3"), w, batch, 128)
    g.prefill([p.cuda() for p in make_prompts(98, [20 + i for i in range(batch)], vocab)])
    cand = torch.randint(0, vocab, (batch, 16), dtype=torch.int32, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4))
    amax, logits = g.verify(cand, want_logits=True)
    g.poll_status()
    hid = g.get_buffer("H_TREE").view(-1, 256)[:batch * 16].double()
    finite = torch.isfinite(lm).all(dim=1)
    ref = hid @ lm[finite].double().T
    got = logits.view(batch * 16, vocab)
    if bool(finite.any()):
        assert float((got[:, finite].double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())      # float sums of 256 terms
    signed = torch.isinf(lm).any(dim=1)
    assert torch.equal(got[:, signed], (torch.sign(hid[:, 3:4]) * float("inf")).float().expand(-1, int(signed.sum())))
    assert bool(torch.isnan(got[:, torch.isnan(lm).any(dim=1)]).all())
    best = torch.where(torch.isnan(got), torch.full_like(got, -float("inf")), got)
    first = ((best == best.max(dim=-1, keepdim=True).values) & ~torch.isnan(got)).int().argmax(dim=-1)
    assert torch.equal(amax.view(-1).long(), first)
    assert torch.equal(g.verify(cand), amax)
    g.close()
