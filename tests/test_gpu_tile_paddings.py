"""Commits of the tile layout's tensor-core path at the operand paddings whose rings differ: with
three splits a padding of 8, 16, .. 64 rows has its own number of ring slots and accumulators (8/8,
8/8, 8/6, 8/5, 7/4, 6/3, 5/2, 5/2), odd ones among them, which the two MMA issuers take in turns.
Matrices long enough that every CTA goes around its ring several times (gate/up of 8192 x 2048
columns: 27 units a CTA); and blocks of 64 rows whose boundary cuts a sequence. Also the many-row
CUDA-core kernel at the row tiles that its own test leaves out (25..32 and 41..48 rows)."""
import pytest

import test_gpu_commit as tcommit
import test_gpu_linear_rows as trows

pytestmark = pytest.mark.gpu


def _spec(d, H_, Hkv, ffn, B, seed, N, page=0, max_seq=48):
    return dict(d=d, n_heads=H_, n_kv_heads=Hkv, head_dim=128, ffn=ffn, vocab=1501, n_layers=N, dtype="bf16", B=B, prefix=0,
                top_k=4, rope_theta=1e4, seed=seed, page_size=page, max_seq=max_seq)


def _tall(B, seed):
    return _spec(2048, 16, 4, 8192, B, seed, 2), [(7 * b) % 40 for b in range(B)], [1] * B


CASES = {
    "rows20": _tall(20, 31),
    "rows29": _tall(29, 32),
    "rows37": _tall(37, 33),
    "rows45": _tall(45, 34),
    "rows53": _tall(53, 35),
    "rows61": _tall(61, 36),
    # eight sequences of several rows
    "b8_48rows": (_spec(512, 4, 1, 1408, 8, 37, 6), [5, 0, 17, 40, 8, 1, 30, 12], [6] * 8),
    "b7_56rows": (_spec(512, 4, 2, 1408, 7, 38, 8, page=16, max_seq=64), [5, 0, 17, 40, 8, 1, 30], [8] * 7),
    # 79 rows in blocks of 64: sequence 32's rows are 63, 64 and 65
    "b40_cut": (_spec(256, 2, 1, 704, 40, 39, 3, page=8), [(7 * b) % 44 for b in range(40)], [1 + b % 3 for b in range(40)]),
    # 180 rows: three blocks, cuts at rows 64 and 128
    "b60_cuts": (_spec(256, 2, 1, 704, 60, 40, 3), [(11 * b) % 44 for b in range(60)], [3] * 60),
}


@pytest.mark.parametrize("case", list(CASES))
def test_commit(orc, monkeypatch, case):
    import paper_2509_20416_gb300 as fe
    init = fe.fe_draft_init
    # (a handle of 64 sequences keeps the tile layout; 9..32 have a layout of their own)
    monkeypatch.setattr(fe, "fe_draft_init", lambda cfg, W: init(dict(cfg, max_batch=max(cfg["B"], 33 if cfg["B"] > 8 else 8)), W))
    monkeypatch.setenv("FE_DRAFT_TILE_TC", "1")
    monkeypatch.setitem(tcommit.COMMIT, case, CASES[case])
    tcommit.test_commit_parity(orc, case)


ROWS = {
    "b29": (trows._spec(768, 6, 3, 128, 2624, 41), 29),
    "b45": (trows._spec(1024, 8, 1, 128, 1472, 42), 45),
    "b45_two_pass": (trows._spec(4096, 4, 1, 128, 14336, 43, N=1), 45),
}


@pytest.mark.parametrize("case", list(ROWS))
def test_many_rows(monkeypatch, case):
    monkeypatch.setitem(trows.CASES, case, ROWS[case])
    trows.test_bit_identical_to_streaming(monkeypatch, case)
