"""Medusa drafts whose heads share one projection and one candidate pass, at vocabularies of several column blocks and fewer sequences than the
context holds: rows of heads and of their candidate lists against the oracle."""
import pytest

from oracle.hydra_oracle import HydraOracle
from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg
from tests.parity import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("vocab,batch,max_batch,mlp,tree", [(6400, 3, 5, 2, "tree63_d4"), (4224, 1, 2, 3, "tree15_d3"), (2048, 5, 5, 2, "tree63_d4")])
def test_drafts_match_the_oracle(dtype, vocab, batch, max_batch, mlp, tree):
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(1, 256, 2, 128, 512, vocab, dtype=dtype)
    h = HeadCfg(4 if tree == "tree63_d4" else 3, mlp, False, medusa=True)
    w = make_weights(m, h, 99)
    parent = load_tree(tree)
    o = HydraOracle(m, h, parent, w, 160, cache_weights=True)
    g = Hydra(m, h, parent, {k: v.cuda() for k, v in w.items()}, max_batch, 160)
    st = lockstep(o, g, make_prompts(99, [12 + 7 * b for b in range(batch)], vocab), 2, 99)
    assert st.steps == 2
    g.close()
