"""The packed prompt pass of the bfloat16 path (prompts back to back, at most 768 tokens a pass) against the oracle, in lock-step."""
import pytest

from synth import load_tree
from synth.configs import ModelCfg, HeadCfg
from tests.test_gpu_step import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,kv_planes,lens", [
    (128, 2, [512]), (128, 2, [513]), (128, 2, [768]), (128, 2, [769]), (128, 2, [1600]),      # up to one full pass; one row more; several passes
    (128, 2, [700, 67, 1]), (128, 2, [700, 67, 1, 1]), (128, 1, [500, 300, 12, 800]),
    (128, 2, [300, 211, 1, 1, 130, 64]), (128, 1, [500, 12, 1]),         # passes that end inside, at the end of and just after a sequence
    (64, 2, [129, 383, 127]), (64, 1, [1, 511, 2])])
def test_packed_prompt_passes(head_dim, kv_planes, lens):
    m = ModelCfg(2, 256, 256 // head_dim, head_dim, 512, 1024, dtype="bf16", kv_planes=kv_planes)
    st, _ = run(m, HeadCfg(3, 1, True), load_tree("tree15_d3"), lens, 2, 33, max(lens) + 40, kv_layers=(0, 1))
    assert st.steps == 2


@pytest.mark.parametrize("rows", [16, 17, 40, 41, 96, 97])
@pytest.mark.parametrize("d_model", [256, 1280])
def test_row_counts_around_the_norm_clusters(rows, d_model):
    """A pass of few rows shares each row's norm among 8, 4 or 2 CTAs of a cluster, one of many rows does not: the prompt passes at the edges."""
    m = ModelCfg(1, d_model, d_model // 128, 128, 512, 1024, dtype="bf16")
    st, _ = run(m, HeadCfg(1, 1, True), [-1, 0], [rows], 1, 34, rows + 16, kv_layers=(0,))
    assert st.steps == 1
