"""Float path: products with what follows them, in both forms (a warp per column, 32 x 32 tiles) and at their edges, over whole steps against the oracle."""
import pytest

from synth import load_tree
from synth.configs import ModelCfg, HeadCfg
from tests.test_gpu_step import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,head,tree,lens", [
    # widths that are no multiple of a tile (32) or a stage (64 k); rows of 1, 3, 15, 48 and, in a prompt chunk, 192
    ((2, 192, 3, 64, 340, 644), (3, 1, False), "tree15_d3", [70, 1, 33]),
    # two warps a pair of columns (d above 256), tiles in all products of 5 x 64 rows, prefix layer, three-layer heads
    ((2, 512, 4, 128, 1000, 1028), (4, 3, True), "tree63_d4", [70, 20, 64, 9, 65]),
    # draft rows (33 and 30) in tiles, blocks of the gathered rows across their stages
    ((1, 2112, 33, 64, 132, 512), (4, 2, False), "tree63_d4", [5, 9, 20]),
    # Medusa heads
    ((2, 256, 2, 128, 688, 2052), (4, 2, False, True, True), "tree15_d3", [17, 40]),
])
def test_steps_against_the_oracle(model, head, tree, lens):
    st, _ = run(ModelCfg(*model, dtype="fp32"), HeadCfg(*head), load_tree(tree), lens, 3, 83, 160, norm_gain_std=0.1)
    assert st.steps == 3
    # rounded at 24 bits: each product and norm adds about 1e-7, and a layer amplifies what comes in by a small factor (heads: several times a layer)
    assert st.max_hidden_err < 2e-5 and st.max_logit_err < 1e-3 and st.max_hprime_err < 1e-4
