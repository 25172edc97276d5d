"""Single kernels at the edges of their tiles, against the oracle on the same seeded inputs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import paper_2509_05165_b200 as kvc
from paper_2509_05165_b200 import workloads as W
from paper_2509_05165_b200.binding import alloc_outputs

import parity as Pz


def _setup(cfg, **desc_kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    return dev, W.make_workload(cfg, dev), kvc.desc_from_config(cfg, **desc_kw)


@pytest.mark.parametrize("N", [1, 63, 129, 1030])
@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 128), ("f32", 64), ("f32", 128)])
def test_value_norms_at_tile_edges(dtype, d, N):
    """One row, a CTA's rows less and more than full, and several CTAs, for every row width."""
    import oracle
    cfg = W.WorkloadConfig("norm_edges", 2, 4, 2, d, N, 1, batch=2, dtype=dtype, elem_std=1.0, n_sinks=min(4, N), hh_frac=0.0)
    dev, wl, desc = _setup(cfg)
    out = alloc_outputs(desc, 1, wl.k[0].dtype, dev)
    kvc.kvc_score_weighted(desc, wl.q, wl.k, wl.v, out.scores, out.workspace)
    torch.cuda.synchronize()
    S = out.scores.cpu().numpy()
    for l in range(cfg.n_layers):
        for b in range(cfg.batch):
            ref = oracle.score_layer_vnorm(Pz.to_f32_numpy(wl.q[l][b]), Pz.to_f32_numpy(wl.k[l][b]), Pz.to_f32_numpy(wl.v[l][b]),
                                           1.0 / np.sqrt(d), desc.q_pos0, desc.agg_task, desc.agg_group, bool(desc.augment_head_mean))
            Pz.assert_scores_close(S[l, b], ref)
