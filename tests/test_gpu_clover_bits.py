"""The clover blocks and the FP32 operator keep their bits.

FP32 results are compared bit for bit between versions of the library, and the FP32
blocks are roundings of the df64 ones: a df64 sum taken in another order is as
accurate, but now and then rounds an FP32 entry the other way.  The digests are
those of the sums in their first order (term by term, real part's product first).

The links are dyadic numbers made from integers, so that every machine feeds the
same bits; they are near the identity but not SU(3), which no step here needs.
"""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = (6, 4, 2, 6)
DIGESTS = {
    "blocks": "a185de020f1c226c9bad59c339bbd322",
    "inverses": "04d412d9e78dee503a623676021d567a",
    "f32": "4156d61942892c8f0e7d84eb58b82510",
    "f32_full": "0a14bff2eb4817feb160b34bc381027a",
}


def _integers(n, seed, bits):
    """n integers of the given bits, centred on 0, from a linear congruential generator."""
    s = np.empty(n, dtype=np.int64)
    v = seed
    for i in range(n):
        v = (v * 6364136223846793005 + 1442695040888963407) & 0xFFFFFFFFFFFFFFFF
        s[i] = (v >> 40) & ((1 << bits) - 1)
    return s - (1 << (bits - 1))


def _complex(shape, seed, bits, scale):
    n = int(np.prod(shape))
    v = _integers(2 * n, seed, bits).astype(np.float64) * scale
    return (v[:n] + 1j * v[n:]).reshape(shape)


def digests():
    """Digest of each output on the dyadic links."""
    import torch

    from paper_2407_08092_gb300 import lqdd
    V = L[0] * L[1] * L[2] * L[3]
    U = _complex((V, 4, 3, 3), 17, 23, 2.0 ** -24) + np.eye(3)
    x = torch.from_numpy(_complex((V, 4, 3), 18, 23, 2.0 ** -20)).cuda()
    ctx = lqdd.lq_create(lqdd.make_lattice(L, -1, 0.05, 1.0), torch.cuda.current_stream().cuda_stream)
    out = {}
    try:
        lqdd.lq_set_gauge(ctx, torch.from_numpy(U).cuda())
        for name, op, prec in (("blocks", lqdd.LQ_OP_EE, lqdd.LQ_DF64), ("inverses", lqdd.LQ_OP_OO_INV, lqdd.LQ_DF64),
                               ("f32", lqdd.LQ_OP_SCHUR, lqdd.LQ_F32), ("f32_full", lqdd.LQ_OP_FULL, lqdd.LQ_F32)):
            v = x if op == lqdd.LQ_OP_FULL else x[:V // 2].contiguous()
            y = torch.empty_like(v)
            lqdd.lq_apply(ctx, op, prec, v, y)
            got = y.cpu().numpy()
            assert np.isfinite(got).all()
            out[name] = hashlib.sha256(np.ascontiguousarray(got).tobytes()).hexdigest()[:32]
    finally:
        lqdd.lq_destroy(ctx)
    return out


def test_clover_and_f32_outputs_keep_their_bits():
    assert digests() == DIGESTS
