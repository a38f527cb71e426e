"""The slab merge with NaN logits (rows of the LM head that hold one): they are never candidates, and
the finite ones that reach the merge are selected as without them, also when most slabs' best
entry is a NaN. (Within a slab a NaN that comes first stays at the head of the slab's list, whose
finite candidates then fill only the places after it; so the finite entries here start a slab, of 24
or 28 entries at this vocabulary size on 152 SMs.)"""
import pytest
import torch

from fe_synth import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 4])
@pytest.mark.parametrize("finite", [(0, 20), (1992, 2012), (4068, 4088)])
def test_nan_rows(finite, k):
    import paper_2509_20416_gb300 as fe
    cfg = wl.make_config(dict(d=256, n_heads=4, n_kv_heads=4, head_dim=64, ffn=256, vocab=4096, n_layers=2, dtype="f32",
                              B=2, prefix=0, top_k=4, rope_theta=1e4, seed=81, page_size=0))
    W = wl.make_weights(cfg)
    lo, hi = finite
    W["lm_head"][:lo] = W["lm_head"][hi:] = float("nan")
    h = fe.fe_draft_init(dict(cfg, max_batch=2), W)
    hid = torch.randn((2, 2, 256), generator=torch.Generator().manual_seed(4))
    out = fe.fe_lm_head_topk_noalloc(h, hid.cuda(), 2, k)
    assert fe.fe_last_device_status(h) == fe.FE_OK
    h.close()
    x = hid.double().transpose(0, 1)  # [B, N, d]
    z = x * torch.rsqrt(x.square().mean(-1, keepdim=True) + cfg["rms_eps"]) * W["final_norm"].double()
    val, idx = torch.topk(z @ W["lm_head"][lo:hi].double().T, k)
    assert torch.equal(out["topk_id"].cpu().long(), idx + lo)
    assert torch.allclose(out["topk_logit"].cpu().double(), val, rtol=1e-4, atol=1e-5)
