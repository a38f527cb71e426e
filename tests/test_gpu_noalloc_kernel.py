"""fe_lm_head_topk_noalloc computes the same bits whichever LM-head kernel the drafts of its handle
take: its softmax statistics are the 16-row kernel's (expf), also for vocabularies whose drafts
run on the wide kernel (2^x, whose lse is a little further from 64 bits)."""
import pytest
import torch

from fe_synth import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,B,k,T", [(6, 1, 8, 0.7), (4, 4, 16, 1.2), (8, 2, 10, 0.0)])
def test_bits_do_not_depend_on_the_drafts_kernel(monkeypatch, N, B, k, T):
    import paper_2509_20416_gb300 as fe
    cfg = wl.make_config(dict(d=512, n_heads=4, n_kv_heads=1, head_dim=128, ffn=64, vocab=78001, n_layers=N, dtype="bf16",
                              B=B, prefix=0, top_k=k, rope_theta=1e4, seed=71, page_size=0))
    W = wl.make_weights(cfg)
    hid = torch.randn((N, B, cfg["d"]), generator=torch.Generator().manual_seed(3)).cuda() * 2
    got = {}
    for force in ("1", "0", None):
        if force is None:
            monkeypatch.delenv("FE_DRAFT_LMHEAD_16ROW")
        else:
            monkeypatch.setenv("FE_DRAFT_LMHEAD_16ROW", force)
        h = fe.fe_draft_init(dict(cfg, max_batch=B), W)
        out = fe.fe_lm_head_topk_noalloc(h, hid, B, k, T)
        got[force] = {x: out[x].clone() for x in ("topk_id", "topk_logit", "topk_prob", "lse")}
        assert fe.fe_last_device_status(h) == fe.FE_OK
        h.close()
    for force in ("0", None):
        for x, t in got["1"].items():
            assert torch.equal(t, got[force][x]), (force, x)
