"""The middle regime of the tree build (boxes of 4097 to 131,072 points, one
cluster of CTAs per box) against the oracle, bit for bit, at the edges of the
regimes and of the clusters' sizes, with heavy ties and for eta-weighted splits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu


def make(kind, n):
    if kind != "ties":
        return inputs.points(kind, n, seed=n)
    x = np.random.default_rng(n).integers(0, 4, size=(n, 3)).astype(float) - 1.5
    x[::5] *= -1.0
    return x


@pytest.mark.parametrize("eta", [1.0, 0.5, 0.0])
@pytest.mark.parametrize("kind,n,levels", [("uniform", 4096, 2), ("uniform", 4097, 2), ("gmm", 16385, 3),
                                           ("ties", 32771, 3), ("plummer", 65537, 3), ("uniform", 131072, 1),
                                           ("uniform", 131073, 2)])
def test_cluster_split_bit_exact(gpu_lib, kind, n, levels, eta):
    fmm = gpu_lib
    x = make(kind, n)
    g = fmm.fmm_plan_tree(fmm.fmm_plan(torch.from_numpy(x).cuda(), levels, 1, 0.5, eta=eta))
    o = oracle.Tree(x, levels, 1, 0.5, eta=eta).tree()
    for k in ("perm", "begin", "count", "lo", "hi"):
        np.testing.assert_array_equal(g[k], o[k], err_msg=k)
