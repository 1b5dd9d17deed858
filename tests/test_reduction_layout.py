"""Which column reductions of a block share a launch, seen without a device: the pass that sizes the arena lays the launches
out and refuses a model (0 bytes) of which one reduction reads what another one of the same launch writes."""
import pytest

from paper_2608_18469_b200 import binding, synth


@pytest.mark.parametrize("dtype, d, heads, seq, batch", [
    ("f32", 64, 1, 1024, 21),        # gradients of 16.5 MB: the bias gradient is a launch of its own, the weight gradient's sum is not
    ("f32", 256, 4, 1024, 8),
    ("f32", 512, 8, 1024, 4),        # two splits
    ("f32", 256, 4, 1024, 4),        # both in the batch
    ("f32", 90, 3, 20, 3),           # no split
    ("bf16", 256, 4, 1024, 8)])
def test_reductions_of_one_launch_do_not_read_one_another(dtype, d, heads, seq, batch):
    assert binding.arena_bytes(synth.lm_spec(2, d, heads, 2 * d, seq, batch, 64, dtype=dtype)) > 0


@pytest.mark.parametrize("spec", [
    synth.config("C1"), synth.config("C3"), synth.mlp_spec(680, 2136, 5, 3001, "relu", "bf16"),
    synth.with_main(synth.ctr_spec(batch=3001, table_rows=2000, tower=(512, 256, 128))),
    synth.mlp_spec(96, 384, 3, 30000, "gelu", "f32"), synth.mlp_spec(128, 256, 3, 512, "gelu", "bf16", head="goodness")],
    ids=["tiny", "ctr", "ragged", "main", "f32_rows30000", "goodness"])
def test_other_models_are_laid_out_too(spec):
    assert binding.arena_bytes(spec) > 0
