"""The bonus draw of fe_verify_sampled against exact arithmetic: distributions of few entries whose
running sum is known as a fraction, with the pick at chosen places of the cluster (first and
last entries of the vocabulary, of its CTAs' and warps' shares) and, in sums that need more than
48 bits, 2^-50 to 2^-52 beside the deviate, where the draw has to tell the sums apart as double
does."""
from fractions import Fraction

import pytest
import torch

import test_gpu_verify_sampled as tv

pytestmark = pytest.mark.gpu

# deviate, entries whose exact sum is just above it (and that float pairs add up to no more
# than the deviate)
FINE = [
    ("0x1.95098ep-1", ["0x1.d0da32p-3", "0x1.b2c62ep-4", "0x1.e1d1f4p-14", "0x1.d4d65ap-2", "0x1.82fffcp-28", "0x1.4p-50"]),
    ("0x1.b01e4ap-1", ["0x1.2a4424p-2", "0x1.872894p-3", "0x1.8ca602p-11", "0x1.719dd2p-2", "0x1.fdfffcp-27", "0x1.2p-49"]),
    ("0x1.86b368p-1", ["0x1.2c8d2ap-2", "0x1.c76e22p-3", "0x1.adc494p-14", "0x1.fa0f70p-3", "0x1.6d7ffcp-27", "0x1.2p-49"]),
    ("0x1.378cc6p-1", ["0x1.b30da0p-3", "0x1.9ad0dap-3", "0x1.65cfa6p-11", "0x1.8eeecep-3", "0x1.67fffcp-29", "0x1.8p-51"]),
]


def _draws(V):
    """(deviate, {entry: probability}) of one vocabulary size."""
    out = []
    last = (V - 10) // 32 * 32  # the last 32 entries with room for ten
    for base in sorted({0, last // 64 * 32, last}):
        for u, ws in FINE:
            p = {base + i: float.fromhex(w) for i, w in enumerate(ws)}
            out.append((float.fromhex(u), {**p, base + 9: 0.0625}))
    share = -(-V // (8 * 512)) * 512  # entries of a CTA
    at = {0, 1, 31, 32, 511, 512, V // 2, V - 2, V - 1}
    at |= {x + y for x in range(0, V, share) for y in (-1, 0)}
    for t in sorted(x for x in at if 0 <= x < V):
        before, after = sorted({t // 3, max(t - 1, 0)} - {t}), sorted({min(t + 1, V - 1), (t + V) // 2} - {t})
        p = {x: 0.125 for x in before + after}
        out.append((0.125 * len(before) + 0.25, {**p, t: 0.5}))
    return out


@pytest.mark.parametrize("V", [33, 1000, 4097, 8191, 32769, 65537, 131072, 131073])
def test_bonus_draw(V):
    draws = _draws(V)
    B = len(draws)
    fe, h = tv._handle(1, V, 1, B)
    # one child, accepted: the bonus comes from its own target distribution
    tree = fe.fe_build_tree(h, torch.zeros(B, dtype=torch.int32, device="cuda"),
                            torch.full((B, 1, 1), 7, dtype=torch.int32, device="cuda"), 1)
    q, p = torch.zeros(B, 1, V), torch.zeros(B, 2, V)
    q[:, 0, 7] = p[:, 0, 7] = 1.0
    u = torch.full((B, 2), 0.5)
    want = []
    for b, (dev, entries) in enumerate(draws):
        run = Fraction(0)
        pick = None
        for x in sorted(entries):
            p[b, 1, x] = entries[x]
            run += Fraction(entries[x])
            if pick is None and Fraction(dev) < run:
                pick = x
        u[b, 1] = dev
        assert float(u[b, 1]) == dev and pick is not None
        want.append(pick)
    got = fe.fe_verify_sampled(h, tree, torch.zeros(B, 1, 1, dtype=torch.int32, device="cuda"), q.cuda(), p.cuda(),
                               u.cuda(), u.cuda(), 1)
    assert fe.fe_last_device_status(h) == fe.FE_OK
    assert got["n_accept"].tolist() == [1] * B
    assert got["bonus"].tolist() == want
    h.close()


def test_no_entry_above_the_deviate():
    """A total below the deviate gives the last token with a positive probability, wherever its
    CTA is."""
    V = 40000
    fe, h = tv._handle(1, V, 1, 3)
    tree = fe.fe_build_tree(h, torch.zeros(3, dtype=torch.int32, device="cuda"),
                            torch.full((3, 1, 1), 7, dtype=torch.int32, device="cuda"), 1)
    q, p = torch.zeros(3, 1, V), torch.zeros(3, 2, V)
    q[:, 0, 7] = p[:, 0, 7] = 1.0
    for b, x in enumerate((5, 20001, V - 1)):
        p[b, 1, 3], p[b, 1, x] = 0.5, 0.25
    u = torch.full((3, 2), 0.75)
    got = fe.fe_verify_sampled(h, tree, torch.zeros(3, 1, 1, dtype=torch.int32, device="cuda"), q.cuda(), p.cuda(),
                               u.cuda(), u.cuda(), 1)
    assert fe.fe_last_device_status(h) == fe.FE_OK
    assert got["bonus"].tolist() == [5, 20001, V - 1]
    h.close()
