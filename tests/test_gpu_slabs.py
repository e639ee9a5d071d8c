"""Attention layers of rows that take more than one vector per lane (columns in slabs, each weighing the producers anew) and the
half-scores of heads whose vectors are a power of two, a multiple of one, or more than a row group has lanes."""
import numpy as np
import pytest

from workloads import dags
import gpu_util

pytestmark = pytest.mark.gpu


def _star(rng, m, n):
    """Node n - 1 reads all others (more than a block's cached producers), the others a few."""
    g = dags.random_dag(rng, n, m["T"], 8, m["dtype"] == "bf16", window=6)
    keep = g["edge_dst"] != n - 1
    g["edge_src"] = np.concatenate([g["edge_src"][keep], np.arange(n - 1, dtype=np.int32)])
    g["edge_dst"] = np.concatenate([g["edge_dst"][keep], np.full(n - 1, n - 1, np.int32)])
    return g


@pytest.mark.parametrize("H,K,dtype", [(512, 1, "bf16"), (512, 16, "bf16"), (480, 4, "bf16"), (416, 2, "bf16"), (288, 1, "bf16"),
                                       (96, 1, "bf16"), (512, 1, "fp32"), (512, 64, "fp32"), (416, 13, "fp32"), (384, 2, "fp32"),
                                       (160, 4, "fp32"), (192, 1, "fp32")])
@pytest.mark.parametrize("nodes", [1, 33, 300])
def test_rows_of_several_vectors_per_lane(xo, H, K, dtype, nodes):
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3)
    rng = dags.make_rng(H + K + nodes)
    graphs = [dags.random_dag(rng, nodes, m["T"], 8, dtype == "bf16", window=6), _star(rng, m, nodes + 1),
              dags.random_dag(rng, 1, m["T"], 8, dtype == "bf16")]
    batch = dags.flatten(graphs, [0, 3], 3)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 5)
    got = gpu_util.run_gpu(batch, blob)
    want = xo.forward(m, blob, batch)
    for k in ("emb", "probs", "value"):
        gpu_util.assert_close(got[k], want[k], dtype, k)


@pytest.mark.parametrize("H,K", [(288, 3), (320, 8), (384, 4), (480, 2), (512, 1), (512, 8), (512, 64)])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_infinite_feature_in_rows_of_several_vectors_per_lane(xo, H, K, dtype):
    """One infinite shape feature: rows of the layers that are no numbers leave their ReLU as 0, as in the definition (a ReLU
    that kept them made the graph's embedding 0)."""
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3)
    rng = dags.make_rng(H + K)
    graphs = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) for n in (33, 40, 36, 1, 35)]
    graphs[2]["shape"][5, 3] = np.inf
    batch = dags.flatten(graphs, [0, 3, 5], 3)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 5)
    got = gpu_util.run_gpu(batch, blob)
    want = xo.forward(m, blob, batch)
    assert np.linalg.norm(want["emb"][2]) > 0.1 and np.isfinite(want["emb"]).all()
    for k in ("emb", "probs", "value"):
        gpu_util.assert_close(got[k], want[k], dtype, k)
