"""Eq. 8 and the heads where one CTA takes several graphs: graph counts on either side of every such line, hidden widths
that leave partial passes, and an embedding buffer that is not 16-byte aligned."""
import numpy as np
import pytest

from workloads import configs, dags
import gpu_util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("envs,cands,H,Hm,Hm2", [(1, 148, 64, 40, 0), (3, 98, 128, 1, 0), (2, 250, 96, 257, 9),
                                                 (5, 240, 32, 70, 33), (40, 60, 256, 256, 64), (150, 1, 64, 64, 0),
                                                 (1, 1100, 512, 300, 0)])
@pytest.mark.parametrize("dtype", ["fp32"])
def test_many_graphs(xo, envs, cands, H, Hm, Hm2, dtype):
    import torch
    import paper_2304_14698_b200 as xrl
    rng = dags.make_rng(envs + cands)
    m = dict(T=7, S=8, H=H, K=2, L=1, Hm=Hm, Hm2=Hm2, Dg=3, dtype=dtype, A_max=cands + 3)
    graphs, env_off = [], [0]
    for _ in range(envs):
        for _ in range(1 + int(rng.integers(max(0, cands - 2), cands + 1))):
            graphs.append(dags.random_dag(rng, int(rng.integers(1, 6)), m["T"], 8, dtype == "bf16", window=4))
        env_off.append(len(graphs))
    batch = dags.flatten(graphs, env_off, m["A_max"])
    batch["mask"][0, 0] = 0
    batch["model"] = m
    blob, _ = gpu_util.default_weights(batch, 21)
    g0 = rng.normal(size=(len(graphs), 3))
    st, packed = xo.pack(batch)
    assert st == 0
    want = xo.encode(m, blob, batch, packed, g0=g0)
    ag = gpu_util.make_agent(batch)
    try:
        ag.set_weights(blob)
        ag.pack(batch)
        buf = torch.zeros(len(graphs) * H + 4, device="cuda")
        mask = torch.from_numpy(batch["mask"]).cuda()
        for shift in (0, 1):
            emb = buf[shift:shift + len(graphs) * H].view(len(graphs), H)
            probs = torch.empty((envs, m["A_max"] + 1), device="cuda")
            value = torch.empty(envs, device="cuda")
            xrl.xrl_encode(ag.ctx, ag.batch, emb, torch.from_numpy(g0.astype(np.float32)).cuda())
            xrl.xrl_policy_value(ag.ctx, ag.batch, emb, mask, probs, value)
            torch.cuda.synchronize()
            assert ag.device_status() == 0
            gpu_util.assert_close(emb.cpu().numpy(), want["emb"], dtype, "emb")
            st, _, p, v = xo.policy_value(m, blob, batch, want["emb"])
            assert st == 0
            gpu_util.assert_close(probs.cpu().numpy(), p, dtype, "probs")
            gpu_util.assert_close(value.cpu().numpy(), v, dtype, "value")
            assert np.all(probs.cpu().numpy()[p == 0] == 0)
    finally:
        ag.close()
