"""Infinities and values next to them in the three-split tensor-core products (bf16 handles of up to
8 sequences): they come out as the float32 products of the CUDA cores give them."""
import pytest
import torch

from fe_synth import workloads as wl

pytestmark = pytest.mark.gpu

F = 5632  # W_down at d = 1024: four or five 64-column blocks a CTA


def _hidden(monkeypatch, edit, seed):
    """The last hidden states [B, d] of a one-layer draft with edited weights and inputs, on the
    CUDA cores and on the tensor cores."""
    import paper_2509_20416_gb300 as fe
    B = 8
    cfg = wl.make_config(dict(d=1024, n_heads=4, n_kv_heads=1, head_dim=128, ffn=F, vocab=1501, n_layers=1, dtype="bf16",
                              B=B, prefix=20, top_k=4, rope_theta=1e4, seed=seed, page_size=0))
    W, I = wl.make_weights(cfg), wl.make_inputs(cfg)
    ks, vs = wl.make_caches(cfg)
    edit(W, I)
    got = []
    for force in ("0", "1"):
        monkeypatch.setenv("FE_DRAFT_TILE_TC", force)
        h = fe.fe_draft_init(dict(cfg, max_batch=B), W)
        out = torch.empty((1, B, cfg["d"]), device="cuda")
        fe.fe_draft_forward(h, I["feat"].cuda(), I["next_tok"].cuda(), I["prefix_len"].cuda(), [k.cuda() for k in ks],
                            [v.cuda() for v in vs], 4, dbg_hidden=out)
        assert fe.fe_last_device_status(h) == fe.FE_OK
        h.close()
        got.append(out[0].cpu())
    return got


@pytest.mark.parametrize("at", [0, 200, 2900, F - 1])  # at several places of a CTA's blocks of W_down
def test_infinite_activation(monkeypatch, at):
    """gate = 2^60 u_3 and up = 2^80 u_3: the activation overflows in the sequences with u_3 > 0
    (silu of the others' gate is 0), whose hidden states take the sign of their weight."""
    def edit(W, I):
        L = W["layers"][0]
        L["w_gate"][at], L["w_up"][at] = 0, 0
        L["w_gate"][at, 3], L["w_up"][at, 3] = 2.0 ** 60, 2.0 ** 80
        L["w_down"][:, at] = torch.where(L["w_down"][:, at] == 0, 0.01, L["w_down"][:, at])

    cuda, tensor = _hidden(monkeypatch, edit, 91)
    assert not cuda.isnan().any() and cuda.isinf().any() and cuda.isfinite().any()
    assert torch.equal(cuda.isfinite(), tensor.isfinite())
    assert torch.equal(cuda[cuda.isinf()], tensor[cuda.isinf()])
    fin = cuda.isfinite()
    assert torch.allclose(cuda[fin], tensor[fin], rtol=0, atol=2e-5 * cuda[fin].abs().max().item())


@pytest.mark.parametrize("at", [0, 300, 1023])
def test_finite_activation_that_rounds_to_infinity(monkeypatch, at):
    """g = W_fuse feat is (2 - 2^-13) 2^127 in one element (above the largest bf16 by more than half
    a unit) and 0 in the others; x0 = W_in g is finite, its RMSNorm scale 0, so the hidden
    states are x0."""
    def edit(W, I):
        W["w_fuse"][:] = 0
        W["w_fuse"][at, 0] = (2 - 2.0 ** -6) * 2.0 ** 63
        I["feat"][:] = 0
        I["feat"][:, 0] = (1 + 2.0 ** -7) * 2.0 ** 64

    cuda, tensor = _hidden(monkeypatch, edit, 92)
    assert cuda.isfinite().all() and cuda.abs().max() > 1e36
    assert tensor.isfinite().all()
    assert torch.allclose(cuda, tensor, rtol=0, atol=2e-5 * cuda.abs().max().item())


@pytest.mark.parametrize("at", [0, 2900])
def test_nan_activation(monkeypatch, at):
    """A NaN in one MLP activation reaches every hidden state."""
    def edit(W, I):
        W["layers"][0]["w_up"][at, 3] = float("nan")

    cuda, tensor = _hidden(monkeypatch, edit, 93)
    assert cuda.isnan().all() and tensor.isnan().all()
