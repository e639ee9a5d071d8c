"""The tensor-core kernels of Eq. 6 and of the node transform at every hidden width they are built for: widths that end
inside a 64-column chunk, widths above 256 (column slices), heads that cross a slice's end, row counts around a tile."""
import pytest

from workloads import configs, dags
import gpu_util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,K", [(32, 2), (64, 1), (96, 3), (160, 4), (192, 6), (224, 7), (288, 3), (320, 8), (352, 1),
                                 (384, 3), (416, 13), (448, 7), (480, 2), (512, 8), (512, 2)])
@pytest.mark.parametrize("nodes", [1, 127, 129])
def test_bf16_widths(xo, H, K, nodes):
    import paper_2304_14698_b200 as xrl
    rng = dags.make_rng(H + nodes)
    m = dict(T=21, S=8, H=H, K=K, L=2, Hm=24, Dg=1, dtype="bf16", A_max=2)
    graphs = [dags.random_dag(rng, n, m["T"], 8, True) for n in (nodes, 1)]
    batch = dags.flatten(graphs, [0, 2], 2)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 3)
    st, packed = xo.pack(batch)
    assert st == 0
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        for layer in range(m["L"] + 1):
            got = xrl.xrl_debug_node_features(ag.ctx, ag.batch, layer, H)
            want = xo.encode(m, blob, batch, packed, dump_layer=layer, want_nodes=True)
            gpu_util.assert_close(got, want["nodes"], "bf16", f"nodes after stage {layer}")
        assert ag.device_status() == 0
    finally:
        ag.close()


@pytest.mark.parametrize("T", [21, 32, 88, 89, 96])
@pytest.mark.parametrize("H", [32, 64, 96, 160, 192, 224, 320, 512])
def test_bf16_node_update_keeps_every_bit_of_the_edge_sum_and_of_the_bias(H, T):
    """Eq. 6 where all but 2^-19 cancels: an edge sum of 1 + 2^-9 + 2^-19 (20 bits) against the node's own features in the even
    columns, one of 1 + 2^-9 + 2^-18 in a second node against a bias of -(1 + 2^-9 + 2^-19) in the odd ones.  The operands
    are exact, so is every partial sum in fp32: the result is 2^-19 exactly."""
    import numpy as np
    import paper_2304_14698_b200 as xrl
    m = dict(T=T, S=8, H=H, K=1, L=0, Hm=8, Dg=1, dtype="bf16", A_max=1)
    shape = np.zeros((6, 8), np.float32)
    shape[:4, 0] = [1, 2.0**-9, 2.0**-19, 2.0**-18]
    shape[4, :2] = [1, 2.0**-9]
    g = dict(op=np.array([0, 1, 2, 3, T - 1, T - 1], np.int32), shape=shape,
             edge_src=np.array([0, 1, 2, 0, 1, 3], np.int32), edge_dst=np.array([4, 4, 4, 5, 5, 5], np.int32))
    batch = dags.flatten([g], [0, 1], 1)
    batch["model"] = m
    W0, b0 = np.zeros((16 + T, H), np.float32), np.zeros(H, np.float32)
    W0[0] = 1
    W0[8 + T:10 + T, ::2] = -1
    b0[1::2] = -(1 + 2.0**-9 + 2.0**-19)
    ag = gpu_util.make_agent(batch)
    try:
        blob = np.zeros(xrl.xrl_weights_size(ag.ctx) // 4, np.float32)
        blob[:W0.size + H] = np.concatenate([W0.ravel(), b0])
        ag.set_weights(blob)
        ag.pack(batch)
        h = xrl.xrl_debug_node_features(ag.ctx, ag.batch, 0, H)
        assert ag.device_status() == 0
        assert (h[4, ::2] == 2.0**-19).all()
        assert (h[5, 1::2] == 2.0**-19).all()
    finally:
        ag.close()


@pytest.mark.parametrize("H,K", [(64, 2), (192, 6), (320, 2)])
def test_bf16_widths_with_many_tiles_per_cta(xo, H, K):
    """Output tiles with an odd number of 64-column chunks, several tiles per CTA: the staging buffers of one tile's last
    store and the next tile's first must not be the same."""
    import paper_2304_14698_b200 as xrl
    rng = dags.make_rng(H)
    m = dict(T=21, S=8, H=H, K=K, L=1, Hm=24, Dg=1, dtype="bf16", A_max=64)
    g = dags.random_dag(rng, 1500, m["T"], 8, True)
    batch = dags.flatten([g] * 50, [0, 50], 64)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 4)
    one = dags.flatten([g], [0, 1], 64)
    st, packed = xo.pack(one)
    assert st == 0
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        for layer in (0, 1):
            got = xrl.xrl_debug_node_features(ag.ctx, ag.batch, layer, H).reshape(50, 1500, H)
            want = xo.encode(m, blob, one, packed, dump_layer=layer, want_nodes=True)["nodes"]
            for i in range(50):
                gpu_util.assert_close(got[i], want, "bf16", f"copy {i} after stage {layer}")
                assert (got[i] == got[0]).all()
    finally:
        ag.close()


@pytest.mark.parametrize("H,K", [(32, 4), (64, 1), (96, 3), (128, 16), (192, 6), (192, 1), (256, 8), (256, 2)])
@pytest.mark.parametrize("copies", [6, 30])
def test_fp32_widths_on_many_rows(xo, H, K, copies):
    """The split-operand transform (8,192 rows and more): widths with one and several column slices, heads within a slice and
    across, a last tile of 40 or 72 rows, one and several tiles per CTA."""
    import paper_2304_14698_b200 as xrl
    rng = dags.make_rng(H + K)
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=24, Dg=1, dtype="fp32", A_max=64)
    n = 1372
    g = dags.random_dag(rng, n, m["T"], 8)
    batch = dags.flatten([g] * copies, [0, copies], 64)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 4)
    one = dags.flatten([g], [0, 1], 64)
    st, packed = xo.pack(one)
    assert st == 0
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        for layer in (1, 2):
            got = xrl.xrl_debug_node_features(ag.ctx, ag.batch, layer, H).reshape(copies, n, H)
            want = xo.encode(m, blob, one, packed, dump_layer=layer, want_nodes=True)["nodes"]
            # every copy against the definition (the attention kernel takes producers singly or in pairs as a copy's rows
            # fall into its blocks, so copies agree within the fp32 bound, not bit for bit)
            for i in range(copies):
                gpu_util.assert_close(got[i], want, "fp32", f"copy {i} after stage {layer}")
        assert ag.device_status() == 0
    finally:
        ag.close()


@pytest.mark.parametrize("H,K", [(32, 2), (64, 2), (96, 3), (128, 4), (160, 5), (192, 6), (224, 7), (256, 4), (320, 5)])
def test_fp32_transform_of_many_rows_keeps_fp32_accuracy(xo, H, K):
    """Both split-operand products (8,192 rows and more) against 64 bits.  Their sums take 3 H / 8 steps, each cut at the 24th
    bit of a running sum that is half its final size on average: (3 H / 16) 2^-24 of the result, and 4 x 2^-24 for Eq. 6,
    the softmax and the weighted sum.  One dropped part of an operand is 2^-12 of a product and far outside."""
    import numpy as np
    import paper_2304_14698_b200 as xrl
    m = dict(T=9, S=8, H=H, K=K, L=1, Hm=24, Dg=1, dtype="fp32", A_max=64)
    n, copies = 1372, 6
    g = dags.random_dag(dags.make_rng(H), n, m["T"], 8)
    batch = dags.flatten([g] * copies, [0, copies], 64)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 4)
    one = dags.flatten([g], [0, 1], 64)
    st, packed = xo.pack(one)
    assert st == 0
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        got = xrl.xrl_debug_node_features(ag.ctx, ag.batch, 1, H).reshape(copies, n, H)
        want = np.asarray(xo.encode(m, blob, one, packed, dump_layer=1, want_nodes=True)["nodes"], np.float64)
        for i in range(copies):
            assert np.linalg.norm(got[i] - want) <= (3 * H / 16 + 4) * 2.0**-24 * np.linalg.norm(want)
        assert ag.device_status() == 0
    finally:
        ag.close()


@pytest.mark.parametrize("H,K", [(128, 1), (128, 2), (128, 4), (128, 8), (256, 1), (256, 2), (256, 4), (256, 8), (256, 16)])
@pytest.mark.parametrize("nodes", [1, 127, 129])
@pytest.mark.parametrize("fused", [True, False])
def test_bf16_heads_of_every_width(xo, monkeypatch, H, K, nodes, fused):
    """The transform's epilogue at 128 and 256 columns: heads of 32 and 64 columns leave in pieces, the others one by one, a
    head of the whole width keeps the columns with one group of warps."""
    import paper_2304_14698_b200 as xrl
    if not fused:
        monkeypatch.setenv("XRL_NO_FUSED_LAYERS", "1")
    rng = dags.make_rng(H + nodes + K)
    m = dict(T=21, S=8, H=H, K=K, L=2, Hm=24, Dg=1, dtype="bf16", A_max=2)
    batch = dags.flatten([dags.random_dag(rng, n, m["T"], 8, True) for n in (nodes, 1)], [0, 2], 2)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 3)
    st, packed = xo.pack(batch)
    assert st == 0
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        for layer in range(m["L"] + 1):
            got = xrl.xrl_debug_node_features(ag.ctx, ag.batch, layer, H)
            want = xo.encode(m, blob, batch, packed, dump_layer=layer, want_nodes=True)
            gpu_util.assert_close(got, want["nodes"], "bf16", f"nodes after stage {layer}")
        assert ag.device_status() == 0
    finally:
        ag.close()


@pytest.mark.parametrize("H,K", [(64, 1), (128, 1), (256, 1), (32, 2), (96, 3), (160, 4), (192, 3), (224, 7), (512, 4)])
def test_bf16_heads_that_two_groups_of_epilogue_warps_cannot_halve(xo, H, K):
    """64, 128 and 256 columns with one head: a group takes every other tile (three or four tiles per CTA, so both numbers of
    turns); the other widths leave all tiles to one group."""
    test_bf16_widths_with_many_tiles_per_cta(xo, H, K)
