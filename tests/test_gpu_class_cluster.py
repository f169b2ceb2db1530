"""The tree kernel with one CTA per problem and with clusters of 2, 4 and 8, at the batch sizes where the rule changes."""
import pytest

import workloads as W
from test_gpu_class import _solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,B", [(511, 3), (512, 14), (512, 15), (515, 29), (512, 30), (520, 74), (512, 75)])
def test_cluster_sizes(R, B):
    _solve(W.cost_matrix(R, 8, (0.0, 1.0, 6.0, 16.0), 4), B, 0.9, 33)
