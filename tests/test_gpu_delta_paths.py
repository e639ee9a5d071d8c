"""Delta encoding's levels by graph (shared memory) and, for a graph beyond that, pass by pass: both give the full encoder's
embeddings, and the same number of reached rows per layer."""
import numpy as np
import pytest

from workloads import dags
import gpu_util

pytestmark = pytest.mark.gpu


def _run(m, graphs, env_off, blob):
    import torch
    import paper_2304_14698_b200 as xrl
    batch = dags.flatten(graphs, env_off, m["A_max"])
    batch["model"] = m
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        full = torch.empty((len(graphs), m["H"]), device="cuda")
        delta = torch.empty_like(full)
        xrl.xrl_encode(ag.ctx, ag.batch, full)
        xrl.xrl_encode_delta(ag.ctx, ag.batch, torch.from_numpy(batch["base_id"]).cuda(), delta)
        torch.cuda.synchronize()
        assert ag.device_status() == 0
        return full.cpu().numpy(), delta.cpu().numpy(), xrl.xrl_delta_rows(ag.ctx, m["L"])
    finally:
        ag.close()


@pytest.mark.parametrize("nodes", [2, 31, 257, 3000])
@pytest.mark.parametrize("L", [0, 1, 5])
def test_levels_by_graph_and_pass_by_pass(nodes, L):
    m = dict(T=11, S=8, H=64, K=2, L=L, Hm=16, Dg=1, dtype="fp32", A_max=8)
    rng = dags.make_rng(nodes + L)
    graphs, env_off = [], [0]
    for _ in range(2):
        cur = dags.random_dag(rng, max(8, nodes), m["T"], 8, window=6)
        graphs += [cur] + [dags.local_rewrite(rng, cur, m["T"]) for _ in range(4)]
        env_off.append(len(graphs))
    blob, _ = gpu_util.default_weights({"model": m, "n_nodes": np.array([max(8, nodes)])}, 6)
    full, delta, rows = _run(m, graphs, env_off, blob)
    gpu_util.assert_close(delta, full, "fp32", "by graph")
    # the same environments beside one whose graph is too large for the per-graph kernel
    big = dags.random_dag(rng, 16385, m["T"], 8, window=6)
    full2, delta2, rows2 = _run(m, graphs + [big], env_off + [len(graphs) + 1], blob)
    gpu_util.assert_close(delta2, full2, "fp32", "pass by pass")
    assert [r + 16385 for r in rows] == rows2


@pytest.mark.parametrize("nodes,copies", [(2048, 2), (2049, 2), (9777, 2), (9830, 2), (16384, 2), (4096, 255), (4097, 255),
                                          (4096, 254)])
def test_levels_at_the_lines_between_the_two(nodes, copies):
    """Graphs at and beyond the sizes up to which a CTA takes a graph (fewer nodes for few graphs), and sizes whose shared
    memory at five bytes a node would need the opt-in: valid batches all, whichever kernels take them."""
    m = dict(T=11, S=8, H=32, K=2, L=2, Hm=16, Dg=1, dtype="fp32", A_max=copies)
    cur = dags.random_dag(dags.make_rng(nodes), nodes, m["T"], 8, window=6)
    graphs = [cur]
    for c in range(copies):                             # a candidate of the same size: one operator changed
        op = cur["op"].copy()
        i = 1 + c * (nodes // copies)
        op[i] = (op[i] + 1) % m["T"]
        graphs.append(dict(cur, op=op, twin=np.arange(nodes, dtype=np.int32)))
    blob, _ = gpu_util.default_weights({"model": m, "n_nodes": np.array([nodes])}, 6)
    full, delta, rows = _run(m, graphs, [0, len(graphs)], blob)
    gpu_util.assert_close(delta, full, "fp32", "by graph, or pass by pass")
    assert nodes < rows[0] <= rows[1] <= rows[2] < nodes * (1 + copies / 2)
    big = dags.random_dag(dags.make_rng(1), 16385, m["T"], 8, window=6)
    full2, delta2, rows2 = _run(m, graphs + [big], [0, len(graphs), len(graphs) + 1], blob)
    gpu_util.assert_close(delta2, full2, "fp32", "pass by pass")
    assert [r + 16385 for r in rows] == rows2


@pytest.mark.parametrize("extra", [1, 3])
def test_batch_with_edges_on_an_empty_graph(extra):
    """A graph without nodes that was given edges is reported; its slots fall into the last row of the graph before it, whose
    node can then look like its twin by its number of producers.  Delta encoding of such a batch stays inside its arrays and
    gives what the full encoder gives."""
    import torch
    import paper_2304_14698_b200 as xrl
    m = dict(T=11, S=8, H=64, K=2, L=3, Hm=16, Dg=1, dtype="fp32", A_max=4)
    rng = dags.make_rng(40 + extra)
    n = 300
    cur = dags.random_dag(rng, n, m["T"], 8, window=6)
    last = np.arange(n - 1 - extra, n - 1, dtype=np.int32)           # the last node reads `extra` nodes for certain
    keep = cur["edge_dst"] != n - 1
    cur["edge_src"] = np.concatenate([cur["edge_src"][keep], last])
    cur["edge_dst"] = np.concatenate([cur["edge_dst"][keep], np.full(extra, n - 1, np.int32)])
    twin = dict(cur, twin=np.arange(n, dtype=np.int32))
    lost = dict(twin, edge_src=cur["edge_src"][:-extra], edge_dst=cur["edge_dst"][:-extra])
    empty = dict(op=np.zeros(0, np.int32), shape=np.zeros((0, 8), np.float32), edge_src=np.zeros(extra, np.int32),
                 edge_dst=np.ones(extra, np.int32), twin=np.zeros(0, np.int32))
    batch = dags.flatten([cur, twin, lost, empty, twin], [0, 5], m["A_max"])
    batch["model"] = m
    blob, _ = gpu_util.default_weights({"model": m, "n_nodes": np.array([n])}, 6)
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        full = torch.empty((5, m["H"]), device="cuda")
        delta = torch.empty_like(full)
        xrl.xrl_encode(ag.ctx, ag.batch, full)
        xrl.xrl_encode_delta(ag.ctx, ag.batch, torch.from_numpy(batch["base_id"]).cuda(), delta)
        torch.cuda.synchronize()
        assert ag.device_status() == 2
        gpu_util.assert_close(delta.cpu().numpy(), full.cpu().numpy(), "fp32", "delta of a bad batch")
        rows = xrl.xrl_delta_rows(ag.ctx, m["L"])
        assert rows == [n + 1] * (m["L"] + 1)            # the current graph and the one row that gained the slots
    finally:
        ag.close()
