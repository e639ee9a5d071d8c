"""Eq. 8's sums fused with the last attention layer of models whose rows share a warp: graphs that begin and end inside, at and
across the blocks of 8, 16 and 32 rows, one-node graphs, graphs without nodes."""
import numpy as np
import pytest

from workloads import dags
import gpu_util

pytestmark = pytest.mark.gpu


def _run(xo, m, sizes, seed):
    m = dict(m, A_max=len(sizes))
    rng = dags.make_rng(seed)
    bf = m["dtype"] == "bf16"
    none = dict(op=np.zeros(0, np.int32), shape=np.zeros((0, 8), np.float32), edge_src=np.zeros(0, np.int32),
                edge_dst=np.zeros(0, np.int32))
    graphs = [dags.random_dag(rng, n, m["T"], 8, bf, window=6) if n else none for n in sizes]
    batch = dags.flatten(graphs, [0, len(graphs)], len(graphs))
    batch["model"] = m
    blob, _ = gpu_util.default_weights(dict(batch, n_nodes=np.maximum(batch["n_nodes"], 1)), 5)
    got = gpu_util.run_gpu(batch, blob)
    want = xo.forward(m, blob, batch)
    for k in ("emb", "probs", "value"):
        gpu_util.assert_close(got[k], want[k], m["dtype"], k)


@pytest.mark.parametrize("H,K,dtype", [(32, 1, "bf16"), (64, 4, "bf16"), (96, 3, "bf16"), (128, 4, "bf16"), (128, 8, "bf16"),
                                       (32, 2, "fp32"), (64, 1, "fp32")])
@pytest.mark.parametrize("sizes", [(1, 1, 1, 1, 1), (8, 8, 16), (7, 9, 1, 0, 15, 33, 2), (0, 5, 0, 300), (3,)])
def test_graphs_around_blocks_of_eight_rows(xo, H, K, dtype, sizes):
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=len(sizes))
    _run(xo, m, sizes, H + len(sizes))


@pytest.mark.parametrize("rows", [47_359, 47_360, 94_719, 94_737])
def test_graphs_around_larger_blocks(xo, rows):
    m = dict(T=9, S=8, H=32, K=2, L=1, Hm=20, Dg=1, dtype="fp32", A_max=16)
    sizes = [4001, 31, 33, 1, 16, 5000, 0, 7]
    _run(xo, m, sizes + [rows - sum(sizes)], rows)
