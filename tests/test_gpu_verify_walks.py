"""fe_verify_sampled against the oracle at the edges of its kernels, on peaked distributions (T = 0.25):
decisions then lie far from their bounds (none of 384 such sequences within the float32 walk's
rounding by the oracle's margins, seeds 201..204), so that all sequences are compared but one at
most, with walks of all lengths and bonus tokens in every CTA of the cluster. (The inputs' last
bits differ between machines, so the count is a bound and no number.)"""
import pytest

import test_gpu_verify_sampled as tv

pytestmark = pytest.mark.gpu

# (B, N, k, V, T, seed, noise sigma of the target's logits)
WALKS = {
    "v33": (16, 2, 4, 33, 0.25, 151, 0.7),
    "v4097": (16, 3, 6, 4097, 0.25, 152, 0.7),
    "v8191": (16, 3, 6, 8191, 0.25, 153, 0.7),
    "v32768": (16, 3, 8, 32768, 0.25, 154, 0.7),
    "v32769": (16, 3, 8, 32769, 0.25, 155, 0.7),
    "v65537": (16, 2, 8, 65537, 0.25, 156, 0.5),
    "v131072": (16, 2, 8, 131072, 0.25, 157, 0.5),
    "v131073": (16, 2, 8, 131073, 0.25, 158, 0.5),
}


@pytest.mark.parametrize("case", list(WALKS))
def test_every_walk(orc, monkeypatch, case):
    monkeypatch.setitem(tv.SYNTH, case, WALKS[case])
    compare = tv._compare
    monkeypatch.setattr(tv, "_compare", lambda *a: compare(*a[:-1], 1))
    tv.test_sampled_verification_matches_oracle(orc, case)
