"""A step whose layers are wide and whose rows are few, against the oracle."""
import pytest

from paper_2405_10951_b200 import synth
from paper_2405_10951_b200.synth import Config

import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 3])
def test_step_of_few_rows_and_wide_layers(batch):
    """Every epilogue of the split few-tile products (float residual stream, GELU with its stored input, GELU derivative) in one step."""
    cfg = Config("mini_wide", 32, 16, 768, 12, 3, 1536, (10,), batch, (1, 2), (), 1, 1, dtype="bf16", seed=6)
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    P.compare_step(cfg, images, labels, task_ids, params, gpu, P.BF16_TOL, P.BF16_EXACT_MARGIN, P.BF16_SCORE_TOL)
