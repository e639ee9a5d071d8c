"""The dense products of the training step's reverse pass at the sizes where their tiles end: widths that are not a
multiple of the tile, row counts around a chunk and past the line from which whole 128-row tiles are used, and a
gradient buffer that is not 16-byte aligned; and its lists by producer, on nodes with more readers or producers than a
warp's list holds."""
import numpy as np
import pytest

from workloads import dags
import gpu_util
from test_gpu_ppo import BF16_ENTRYWISE, GRAD_TOL, _check_grad, _transitions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,K,dtype,nodes", [(32, 2, "fp32", 63), (96, 3, "fp32", 2100), (128, 4, "fp32", 2050),
                                             (160, 4, "fp32", 257), (384, 3, "fp32", 65), (64, 2, "bf16", 127),
                                             (192, 6, "bf16", 2100), (384, 3, "bf16", 65), (128, 4, "bf16", 129),
                                             (256, 8, "bf16", 1), (512, 8, "bf16", 131)])
def test_gradient_at_the_edges_of_the_tiles(xo, H, K, dtype, nodes):
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3)
    rng = dags.make_rng(H + nodes)
    sizes = [nodes, nodes + 3, nodes, 1, nodes + 1]
    graphs = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) for n in sizes]
    _compare(xo, dags.flatten(graphs, [0, 3, 5], 3), m)


def _star(rng, m, readers, producers, repeats):
    """Node 0 is read by `readers` nodes, the last node reads `producers` of them (and node 1 `repeats` times)."""
    n = readers + 2
    src = [0] * readers + list(range(1, producers + 1)) + [1] * repeats
    dst = list(range(1, readers + 1)) + [n - 1] * (producers + repeats)
    g = dags.random_dag(rng, n, m["T"], 8, m["dtype"] == "bf16")
    g["edge_src"], g["edge_dst"] = np.array(src, np.int32), np.array(dst, np.int32)
    return g


@pytest.mark.parametrize("H,K,dtype,both", [(128, 2, "fp32", False), (128, 4, "fp32", False), (128, 16, "fp32", True),
                                            (256, 8, "fp32", False), (128, 8, "bf16", False), (256, 2, "bf16", False),
                                            (256, 4, "bf16", True), (256, 8, "bf16", False), (256, 16, "bf16", False)])
def test_gradient_with_long_lists(xo, H, K, dtype, both):
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3, both_ways=both)
    rng = dags.make_rng(H + K)
    graphs = [_star(rng, m, *v) for v in ((94, 2, 0), (95, 94, 1), (96, 95, 0), (97, 96, 3), (200, 150, 40))]
    _compare(xo, dags.flatten(graphs, [0, 3, 5], 3), m)


def _compare(xo, batch, m):
    import torch
    import paper_2304_14698_b200 as xrl
    dtype = m["dtype"]
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 7)
    st, packed = xo.pack(batch)
    assert st == 0
    action, logp_old, adv, ret = _transitions(xo, m, blob, batch, packed, 5)
    want = xo.ppo_grad(m, blob, batch, packed, action, logp_old, adv, ret)
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        f32 = lambda a: torch.from_numpy(np.asarray(a, np.float32)).cuda()
        buf = torch.full((len(blob) + 4,), 7.0, device="cuda")
        loss = torch.empty(4, device="cuda")
        for shift in (0, 1):
            grad = buf[shift:shift + len(blob)]
            xrl.xrl_ppo_grad(ag.ctx, ag.batch, torch.from_numpy(batch["mask"]).cuda(), torch.from_numpy(action).cuda(),
                             f32(logp_old), f32(adv), f32(ret), loss, grad)
            torch.cuda.synchronize()
            assert ag.device_status() == 0
            gpu_util.assert_close(loss.cpu().numpy(), want["loss"], dtype, "loss")
            _check_grad(m, grad.cpu().numpy().astype(np.float64), want["grad"], GRAD_TOL[dtype], f"shift {shift}",
                        entrywise=BF16_ENTRYWISE if dtype == "bf16" else None)
    finally:
        ag.close()


@pytest.mark.parametrize("H,K,dtype,both,extra", [(128, 4, "fp32", False, 1), (128, 2, "bf16", True, 7),
                                                  (256, 8, "bf16", False, 200), (256, 4, "bf16", True, 200)])
def test_gradient_of_a_batch_whose_first_graph_has_edges_and_no_nodes(H, K, dtype, both, extra):
    """Such a batch is reported; its first slots belong to no row.  The gradient is then that of the batch without them, up to
    the order of its atomic sums (a few thousand fp32 terms: 1e-5 of the gradient)."""
    import torch
    import paper_2304_14698_b200 as xrl
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3, both_ways=both)
    rng = dags.make_rng(H + extra)
    rest = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) for n in (60, 64, 90, 61)]
    got = []
    for k in (extra, 0):
        empty = dict(op=np.zeros(0, np.int32), shape=np.zeros((0, 8), np.float32), edge_src=np.zeros(k, np.int32),
                     edge_dst=np.ones(k, np.int32))
        batch = dags.flatten([empty] + rest, [0, 2, 5], 3)
        batch["model"] = m
        blob, _ = gpu_util.default_weights({"model": m, "n_nodes": np.array([60])}, 7)
        ag = gpu_util.make_agent(batch)
        try:
            ag.set_weights(blob)
            ag.pack(batch)
            f32 = lambda *a: torch.tensor(a, device="cuda")
            grad, loss = torch.empty(len(blob), device="cuda"), torch.empty(4, device="cuda")
            xrl.xrl_ppo_grad(ag.ctx, ag.batch, torch.from_numpy(batch["mask"]).cuda(),
                             torch.tensor([0, 3], dtype=torch.int32, device="cuda"), f32(-0.7, -1.0), f32(1.0, -0.5),
                             f32(0.3, 0.1), loss, grad)
            torch.cuda.synchronize()
            assert ag.device_status() == (2 if k else 0)
            got.append((loss.cpu().numpy(), grad.cpu().numpy().astype(np.float64)))
        finally:
            ag.close()
    np.testing.assert_allclose(got[0][0], got[1][0], rtol=1e-5, atol=1e-6)
    assert np.linalg.norm(got[1][1]) > 0
    assert np.linalg.norm(got[0][1] - got[1][1]) <= 1e-5 * np.linalg.norm(got[1][1])


def test_gradient_where_the_lists_by_producer_do_not_fit():
    """A context whose workspace fits the GPU's free memory without those lists and not with them: the call scatters instead
    of refusing, with the same gradient (fp32 sums in another order: 1e-5)."""
    import torch
    import paper_2304_14698_b200 as xrl
    m = dict(T=9, S=8, H=128, K=16, L=1, Hm=20, Dg=1, dtype="fp32", A_max=3)
    rng = dags.make_rng(8)
    batch = dags.flatten([dags.random_dag(rng, n, m["T"], 8, window=6) for n in (60, 64, 90, 61)], [0, 4], 3)
    blob, _ = gpu_util.default_weights(dict(batch, model=m), 7)
    N, E = 50_000, 6_000_000
    lists = 8 * m["K"] * (N + E)
    f32 = lambda *a: torch.tensor(a, device="cuda")
    mask, action = torch.from_numpy(batch["mask"]).cuda(), torch.tensor([1], dtype=torch.int32, device="cuda")
    logp, adv, ret, loss = f32(-1.0), f32(1.0), f32(0.3), torch.empty(4, device="cuda")
    grads, used, filler = [torch.empty(len(blob), device="cuda") for _ in range(2)], 0, None
    for i in range(2):
        ag = xrl.Agent(m, 4, 1, N, E)
        try:
            ag.set_weights(blob)
            ag.pack(batch)
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            free = torch.cuda.mem_get_info()[0]
            if i:
                filler = torch.empty(free - used + lists // 2, dtype=torch.uint8, device="cuda")
            xrl.xrl_ppo_grad(ag.ctx, ag.batch, mask, action, logp, adv, ret, loss, grads[i])
            torch.cuda.synchronize()
            used = free - torch.cuda.mem_get_info()[0]
            assert ag.device_status() == 0
        finally:
            ag.close()
    del filler
    torch.cuda.empty_cache()
    assert (grads[1] - grads[0]).norm() <= 1e-5 * grads[0].norm() and grads[0].norm() > 0


@pytest.mark.parametrize("H,K,nodes", [(256, 8, 30), (256, 8, 31), (256, 4, 63), (128, 8, 31), (128, 2, 127), (256, 8, 9600)])
def test_gradient_of_both_products_at_the_edges_of_their_tiles(xo, H, K, nodes):
    """125, 129, 257, 513 rows (one to five tiles of 128, one or two CTAs per half) and 38,405 (several tiles per CTA, an odd
    number of rows)."""
    m = dict(T=9, S=8, H=H, K=K, L=1 if nodes > 1000 else 2, Hm=20, Dg=1, dtype="bf16", A_max=3)
    rng = dags.make_rng(H + nodes)
    graphs = [dags.random_dag(rng, n, m["T"], 8, True, window=6) for n in (nodes, nodes + 3, nodes, 1, nodes + 1)]
    _compare(xo, dags.flatten(graphs, [0, 3, 5], 3), m)


def _no_nodes():
    return dict(op=np.zeros(0, np.int32), shape=np.zeros((0, 8), np.float32), edge_src=np.zeros(0, np.int32),
                edge_dst=np.zeros(0, np.int32))


@pytest.mark.parametrize("H,K,dtype,sizes", [
    (H, K, dtype, sizes) for H, K, dtype in ((256, 4, "bf16"), (256, 8, "bf16"), (256, 16, "bf16"), (128, 4, "fp32"),
                                             (128, 8, "fp32"), (128, 4, "bf16"))
    for sizes in ((1, 1, 1, 1), (7, 8, 9, 1, 15, 17), (0, 5, 0, 33), (300, 0, 1, 700))
    if dtype == "fp32" or sum(sizes) > 4])    # (four bf16 nodes: one rounded ReLU is a matrix column)
def test_gradient_of_the_readout_fused_with_the_last_layer(xo, H, K, dtype, sizes):
    """Graphs that begin and end inside, at and across the last layer's blocks of eight rows, graphs without nodes, and more
    graphs than blocks (their sums then do not fit and the readout runs on its own)."""
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=len(sizes))
    rng = dags.make_rng(H + K + len(sizes))
    graphs = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) if n else _no_nodes() for n in sizes]
    _compare(xo, dags.flatten(graphs, [0, len(graphs)], m["A_max"]), m)


def _library_that_declines(name, out):
    """libxrl.so with the launcher `name` replaced by one that declines every call, as it does where a tensor map is refused."""
    import glob
    import os
    import subprocess
    from paper_2304_14698_b200 import build
    sources = [os.path.basename(s)[:-3] for s in sorted(glob.glob(os.path.join(build.CSRC, "*.cu")))]
    objects = [os.path.join(build.OBJ, s + ".o") for s in sources]
    if not all(map(os.path.exists, objects)):
        build.build()
    symbols = subprocess.run(["nm", *objects], capture_output=True, text=True, check=True).stdout.split()
    symbol, = {s for s in symbols if s.startswith(f"_ZN3xrl{len(name)}{name}E")}
    stub, lib = str(out / "stub.cpp"), str(out / "libxrl_declines.so")
    with open(stub, "w") as f:
        f.write(f'extern "C" int __wrap_{symbol}() {{ return -1; }}\n')
    subprocess.run([build._nvcc(), "-shared", "-Xcompiler", "-fPIC", "-o", lib, *objects, stub, "-Xlinker", f"--wrap={symbol}",
                    "-gencode", "arch=compute_100a,code=sm_100a"], check=True)
    return lib


@pytest.mark.parametrize("H,K,dtype", [(256, 8, "bf16"), (128, 4, "fp32")])
def test_gradient_where_the_gather_of_the_softmax_reverse_declines(xo, monkeypatch, tmp_path, H, K, dtype):
    """The kernel without TMA reads rows of gradients, which the last layer then has to have written."""
    from paper_2304_14698_b200 import binding
    monkeypatch.setattr(binding, "_LIB_PATH", _library_that_declines("launch_rows_gather", tmp_path))
    monkeypatch.setattr(binding, "_lib", None)
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3)
    rng = dags.make_rng(H)
    graphs = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) for n in (65, 70, 65, 33, 66)]
    _compare(xo, dags.flatten(graphs, [0, 3, 5], 3), m)


@pytest.mark.parametrize("H,K,dtype,nodes", [
    (H, K, dtype, nodes) for H, K in ((96, 1), (96, 4), (160, 2), (192, 4), (192, 8), (224, 4), (288, 4), (320, 8), (352, 1),
                                      (384, 4), (416, 2), (448, 8), (480, 4))
    for dtype, nodes in (("fp32", 3), ("fp32", 40), ("bf16", 130))] + [(96, 2, "bf16", 2500), (192, 4, "fp32", 2500),
                                                                     (384, 12, "fp32", 40), (192, 12, "bf16", 130)])
def test_gradient_of_widths_without_a_power_of_two(xo, H, K, dtype, nodes):
    """Every number of features per lane that is no power of two (pieces on 2- to 16-byte boundaries): CTAs whose warps have no
    row, one, two, and (10,000 rows) several; then heads that do not divide a warp."""
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype=dtype, A_max=3)
    rng = dags.make_rng(H + K + nodes)
    graphs = [dags.random_dag(rng, n, m["T"], 8, dtype == "bf16", window=6) for n in (nodes, nodes + 3, nodes, 1, nodes + 1)]
    _compare(xo, dags.flatten(graphs, [0, 3, 5], 3), m)


@pytest.mark.parametrize("H,K", [(96, 1), (96, 4), (160, 4), (192, 1), (192, 8), (320, 2), (384, 4), (480, 2)])
def test_gradient_of_an_infinite_feature_shows_it(xo, H, K):
    """One infinite shape feature: the first layer's matrix, attention vectors and Eq. 6's bias have gradients that are no
    numbers where the definition's are (rows and half-scores passed over as zeros gave finite ones)."""
    import torch
    import paper_2304_14698_b200 as xrl
    from workloads import configs
    m = dict(T=9, S=8, H=H, K=K, L=2, Hm=20, Dg=1, dtype="fp32", A_max=3)
    rng = dags.make_rng(H + K)
    graphs = [dags.random_dag(rng, n, m["T"], 8, window=6) for n in (33, 40, 36, 1, 35)]
    graphs[2]["shape"][5, 3] = np.inf
    batch = dags.flatten(graphs, [0, 3, 5], 3)
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 5)
    st, packed = xo.pack(batch)
    assert st == 0
    action, logp, adv, ret = np.array([3, 3], np.int32), np.array([-0.7, -1.0]), np.array([1.0, -0.5]), np.array([0.3, 0.1])
    want = xo.ppo_grad(m, blob, batch, packed, action, logp, adv, ret)["grad"]
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        f32 = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
        grad, loss = torch.empty(len(blob), device="cuda"), torch.empty(4, device="cuda")
        xrl.xrl_ppo_grad(ag.ctx, ag.batch, torch.from_numpy(batch["mask"]).cuda(), torch.from_numpy(action).cuda(), f32(logp),
                         f32(adv), f32(ret), loss, grad)
        got = grad.cpu().numpy()
        assert ag.device_status() == 0
    finally:
        ag.close()
    off, seen = 0, 0
    for name, shape in configs.weight_layout(m):
        part = slice(off, off + int(np.prod(shape)))
        off = part.stop
        if name in ("b0", "W1", "a_src1", "a_dst1"):
            assert np.array_equal(np.isnan(got[part]), np.isnan(want[part])), name
            seen += int(np.isnan(want[part]).sum())
    assert seen > H
