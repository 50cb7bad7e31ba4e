"""Rounds on either side of the lines where the one-launch search changes its blocks: how many candidates share an SM (148
on a B200) and how many jobs keep their records in shared memory.  Bit for bit the dense entry points one by one."""
import pytest

import test_gpu_round_shapes as shapes

pytestmark = pytest.mark.gpu

# as in test_gpu_round_shapes: nodes, GPUs per node, jobs, population, generations, nodes per rack, active, perturbation
KINDS = [
    (20, 4, 256, 148, 4, 0, 1.0, 0.2), (20, 4, 256, 149, 4, 6, 1.0, 0.2), (20, 4, 257, 148, 4, 6, 1.0, 0.2),
    (20, 4, 257, 149, 4, 0, 1.0, 0.2), (12, 8, 1024, 30, 3, 4, 0.8, 0.1), (12, 8, 1025, 30, 3, 0, 1.0, 0.1),
    (12, 8, 700, 296, 3, 0, 1.0, 0.1), (12, 8, 300, 297, 3, 0, 1.0, 0.1), (20, 4, 64, 296, 4, 0, 1.0, 0.2),
    (20, 4, 64, 297, 4, 0, 0.5, 0.2), (20, 4, 64, 445, 4, 5, 1.0, 0.2), (64, 4, 900, 200, 3, 0, 1.0, 0.9),
    (1, 4, 1, 3, 3, 0, 1.0, 1.0),
]


@pytest.mark.parametrize("shape", KINDS, ids=lambda s: "-".join(str(x) for x in s))
@pytest.mark.parametrize("start", ["none", "feasible", "raw"])
def test_rounds_at_the_kinds_edges(shape, start):
    shapes.test_round_equals_stepwise("flow", shape, start)
