"""The residual buffer of fe_verify_sampled: held only by handles whose vocabulary needs it."""
import pytest
import torch

from fe_synth import workloads as wl

pytestmark = pytest.mark.gpu


def _held(V):
    import paper_2509_20416_gb300 as fe
    cfg = wl.make_config(dict(d=64, n_heads=1, n_kv_heads=1, head_dim=64, ffn=64, vocab=V, n_layers=1, dtype="bf16", B=64,
                              prefix=0, top_k=1, rope_theta=1e4, seed=1, page_size=0))
    W = wl.make_weights(cfg)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = fe.fe_draft_init(dict(cfg, max_batch=64), W)
    held = before - torch.cuda.mem_get_info()[0]
    h.close()
    return held


def test_residuals_only_above_the_register_kernel():
    torch.zeros(1, device="cuda")
    _held(1000)  # (what the first handle of a process brings with it)
    small, large = _held(131072), _held(131073)
    assert large - small > 0.8 * 64 * 131073 * 4, (small, large)
