"""Sizes at the edges of the kernels' tiles and dispatch rules, against the oracle or an fp64 restatement of the op."""
import numpy as np
import pytest

from paper_2405_10951_b200 import synth
from paper_2405_10951_b200.synth import Config

import parity as P

pytestmark = pytest.mark.gpu

MINI = Config("mini_shapes", 64, 8, 128, 2, 6, 256, (10,), 6, (3, 4, 5), (1, 3, 4), 7, 10, dtype="bf16", seed=1)


@pytest.mark.parametrize("batch", [1, 3, 5, 7])
def test_bf16_step_with_odd_row_counts(batch):
    """Weight gradients reduce over batch x tokens rows, which no tile divides here; same tolerance as every bf16 step."""
    cfg = MINI.with_(batch=batch, trainable=(1, 3, 5))
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    P.compare_step(cfg, images, labels, task_ids, params, gpu, P.BF16_TOL, P.BF16_EXACT_MARGIN, P.BF16_SCORE_TOL)
