"""Commits whose rows have no place in the cache: the multi-row path (bf16, head size 128, tensor
cores) reports and leaves out what the launch per row does. A sequence without rows to commit is
not looked at, whatever its prefix_len; of a sequence with rows, those at positions in
0 .. max_seq - 1 are stored; a prefix_len at the ends of its type stores nothing."""
import pytest
import torch

from fe_synth import workloads as wl
import harness as H
import test_gpu_commit as tcommit

pytestmark = pytest.mark.gpu

MAX = 2 ** 31 - 1

# prefix lengths, rows to commit, every row has a place, the launch per row is asked too
CASES = {
    # an idle slot far out of range
    "idle_out_of_range": ([5, 49, 1000000, -3], [3, 0, 0, 0], True, True),
    # rows before position 0 and past the last one, in sequences with valid rows besides
    "cut_at_both_ends": ([-1, -2, 46, 45], [4, 2, 4, 3], False, True),
    "ends_of_the_type": ([MAX, MAX - 3, -MAX - 1, 7], [4, 4, 4, 2], False, False),
    "idle_at_the_ends": ([MAX, -MAX - 1, 9, MAX - 7], [0, 0, 4, 0], True, False),
}


@pytest.mark.parametrize("layers", [1, 4])
@pytest.mark.parametrize("case", list(CASES))
def test_rows_without_a_place(monkeypatch, case, layers):
    import paper_2509_20416_gb300 as fe
    P, n, fits, per_row = CASES[case]
    spec = dict(d=256, n_heads=4, n_kv_heads=2, head_dim=128, ffn=704, vocab=1501, n_layers=layers, dtype="bf16", B=4,
                prefix=0, top_k=4, rope_theta=1e4, seed=61, page_size=0, max_seq=48)
    n = [min(x, layers) for x in n]
    cfg = wl.make_config(spec)
    W = wl.make_weights(cfg)
    ks, vs = wl.make_caches(cfg)
    feats = tcommit._feats(cfg, 4, layers, 70)
    toks = torch.randint(0, 1501, (4, layers), generator=torch.Generator().manual_seed(5), dtype=torch.int32)
    got = {}
    # (the launch per row forms prefix_len + row in 32 bits: not asked at the ends of the type)
    for force in ("0", "1") if per_row else ("1",):
        monkeypatch.setenv("FE_DRAFT_TILE_TC", force)
        h = fe.fe_draft_init(dict(cfg, max_batch=4), W)
        kd, vd, _, _ = H.device_caches(cfg, ks, vs, None)
        fe.fe_commit(h, feats.cuda(), toks.cuda(), torch.tensor(n, dtype=torch.int32).cuda(),
                     torch.tensor(P, dtype=torch.int32).cuda(), kd, vd)
        st = fe.fe_last_device_status(h)
        h.close()
        some_out = any(not (0 <= p + i < 48) for p, m in zip(P, n) for i in range(m))
        assert st == (fe.FE_ERR_CAPACITY if some_out else fe.FE_OK), (force, st)
        assert fits is not some_out
        got[force] = [t.cpu() for t in kd + vd]
        # exactly the rows with a place were stored
        for new, old in zip(got[force], list(ks) + list(vs)):
            same = (new == old).all(-1).all(1)  # [B, max_seq]
            for b in range(4):
                rows = {P[b] + i for i in range(n[b])}
                for pos in range(48):
                    assert bool(same[b, pos]) == (pos not in rows), (force, b, pos)
    if per_row:
        for x, y in zip(got["0"], got["1"]):  # one bf16 rounding apart at most
            assert torch.allclose(x.float(), y.float(), rtol=2.0 ** -7, atol=2.0 ** -8)
