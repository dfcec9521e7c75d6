"""The force of a lattice larger than its plaquette scratch goes through the
links in ranges of time slices: with periodic time the gradient of fields
shifted by some slices is the shifted gradient, whichever range a slice falls in.

Each link's sums run over the same numbers in the same order wherever the
range begins, so the two gradients agree bit for bit.
"""
import numpy as np
import pytest

from paper_2407_08092_gb300 import synth

pytestmark = pytest.mark.gpu


def test_force_of_shifted_fields_is_the_shifted_force():
    import torch

    from paper_2407_08092_gb300 import lqdd
    L, shift = (24, 24, 24, 32), 5   # 5184 B x 24^3 a slice: more slices than 2 GiB of scratch hold
    s3 = L[0] * L[1] * L[2]
    U = torch.from_numpy(synth.gauge_links(L, 0.25, 77)).cuda()
    X = torch.from_numpy(synth.gaussian_spinor(s3 * L[3], 78)).cuda()
    Y = torch.from_numpy(synth.gaussian_spinor(s3 * L[3], 79)).cuda()
    ctx = lqdd.lq_create(lqdd.make_lattice(L, 1, 0.05, 1.0), torch.cuda.current_stream().cuda_stream)
    try:
        out = []
        for k in (0, shift):
            def roll(v):
                return torch.roll(v, k * s3, 0).contiguous()
            G = torch.empty_like(U)
            lqdd.lq_set_gauge(ctx, roll(U))
            lqdd.lq_force(ctx, roll(X), roll(Y), G, coef=-2.0)
            out.append(torch.roll(G, -k * s3, 0).cpu().numpy())
        assert np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0
        assert np.array_equal(out[0], out[1])
    finally:
        lqdd.lq_destroy(ctx)
