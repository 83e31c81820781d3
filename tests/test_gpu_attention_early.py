"""Decoding without a tree on the tensor-core path, against the oracle: the one-row attention reads committed keys ahead of its wait, over several rounds of a CTA and
several chunks of a pair (two heads: up to eight)."""
import pytest
import torch

from oracle.hydra_oracle import HydraOracle
from synth import make_weights, make_prompts
from synth.configs import ModelCfg, HeadCfg
from tests.parity import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,planes", [(128, 2), (128, 1), (64, 2), (64, 1)])
@pytest.mark.parametrize("lens", [[130], [520, 64], [1100, 447]])
def test_root_only_steps_over_several_chunks(lens, head_dim, planes):
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(2, 256, 256 // head_dim, head_dim, 512, 1024, dtype="bf16", kv_planes=planes)
    h = HeadCfg(1, 1, True)                                # (the prefix layer takes two rows a step)
    w = make_weights(m, h, 51)
    max_seq = max(lens) + 40
    o = HydraOracle(m, h, [-1], w, max_seq, cache_weights=True)
    g = Hydra(m, h, [-1], {k: v.cuda() for k, v in w.items()}, len(lens), max_seq)
    try:
        st = lockstep(o, g, make_prompts(51, lens, m.vocab), 4, 51, plant=False, kv_layers=(0, 1))
        assert st.steps == 4
    finally:
        g.close()
