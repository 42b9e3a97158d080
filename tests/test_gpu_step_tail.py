"""The step tail's merge warps (one or two query heads per KV head) over every way of merging the partials: a few
per head, up to 32 (one read of the statistics), more than 32. Compared, as in test_gpu_step_fused, with the separate
entry points: the arithmetic and its order are the same, so outputs, scores, victims and demoted rows have to be the
same bits."""
import pytest
import torch

import mikv_inputs as mi
import test_gpu_step_fused as fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [
    mi.Workload("tail1few", 40, 8, 8, 70, 1, 2, 32, 0.2, seed=61),   # G = 1, one or two partials per head
    mi.Workload("tail1mid", 4, 24, 24, 700, 1, 2, 32, 0.2, seed=62),  # G = 1, up to 32
    mi.Workload("tail1many", 1, 1, 1, 9000, 1, 3, 128, 0.05, seed=63),  # G = 1, more than 32
    mi.Workload("tail2few", 30, 8, 4, 130, 1, 4, 64, 0.2, seed=64),  # G = 2
    mi.Workload("tail2mid", 2, 32, 16, 1500, 1, 2, 64, 0.3, seed=65),
    mi.Workload("tail2many", 1, 2, 1, 9000, 1, 2, 32, 0.2, seed=66),
], ids=lambda w: w.name)
def test_merge_warps(w):
    fused.test_fused_step_equals_separate_calls(w, torch.float32)
    fused.test_fused_step_equals_separate_calls(w, torch.bfloat16)
