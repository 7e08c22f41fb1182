"""The grouped launches of the fp32 path over several layers at once, against the float64 oracle, with the tolerance of
the other fp32 parity tests: every tile form, at ragged edges and with one-sided layers of either orientation (the
transposed and plain operands of each form), bf16 and clipped gradients (materialised in fp32), more layers than one
launch takes, layers of a chunk that refresh while others do not.

The form of a launch follows from the number of 32 x 32 tiles of its results, N: up to 592 four groups of threads share
the contraction of a 32 x 32 tile, up to 1776 one does, up to 9472 (and above, in the launch that takes two products
together) 64 x 64 tiles, above 128 x 128.  `launches` are the N of a case's launches: the factors together
with the first sides, and the pairs, back products and weight updates."""
import pytest

from workloads import LayerSpec, Workload
from workloads.configs import GEOM_BI, GEOM_UNI, SRC_FIRST, SRC_SECOND

pytestmark = pytest.mark.gpu
TOL = 1e-4          # relative Frobenius error of an update: fp32 chains of at most 3.4e3 terms through five products


def _layers(shapes, geoms, srcs, tau=1, freqs=(0,)):
    return [LayerSpec("W%d" % i, m, n, geoms[i % len(geoms)], srcs[i % len(srcs)], tau, freqs[i % len(freqs)])
            for i, (m, n) in enumerate(shapes)]


def launches(layers):
    t = lambda m, n: -(-m // 32) * -(-n // 32)
    factors = sum((t(l.m, l.m) if l.geom == GEOM_BI or l.m <= l.n else 0) + (t(l.n, l.n) if l.geom == GEOM_BI or l.m > l.n else 0)
                  for l in layers if l.src == SRC_SECOND)
    return {"factors": factors + sum(2 * t(l.m, l.n) for l in layers if l.geom == GEOM_BI), "rest": sum(t(l.m, l.n) for l in layers)}


CASES = {
    "tiles32_ragged": _layers([(131, 33), (33, 140), (200, 129)], [GEOM_BI, GEOM_UNI], [SRC_SECOND]),
    "tiles32_two_layers": _layers([(1100, 260), (260, 1301)], [GEOM_UNI], [SRC_SECOND]),
    "tiles32_whole": _layers([(801, 700), (700, 333)], [GEOM_UNI], [SRC_SECOND]),
    "tiles64": _layers([(1400, 1300), (130, 3300)], [GEOM_UNI], [SRC_SECOND]),
    "tiles64_both": _layers([(1009, 971), (1001, 1333)], [GEOM_BI, GEOM_UNI], [SRC_SECOND]),
    "many": _layers([(130 + i, 20 + i) for i in range(35)], [GEOM_UNI, GEOM_BI], [SRC_SECOND]),
    "mixed_periods": _layers([(140, 139), (150, 40), (40, 150)], [GEOM_BI, GEOM_UNI], [SRC_SECOND, SRC_FIRST], freqs=(2, 3, 5)),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("grad,clip", [("f32", 0.0), ("bf16", 0.5)])
def test_group(name, grad, clip):
    import paper_2602_03515_b200 as br
    from tests.parity_util import SideBySide, rel_l2
    n = launches(CASES[name])
    if name == "tiles32_ragged":
        assert max(n.values()) <= 592
    elif name == "tiles32_whole":
        assert 592 < min(n.values()) and max(n.values()) <= 1776
    elif name == "tiles64":
        assert 1776 < n["rest"] <= 9472
    elif name == "tiles64_both":
        assert 1776 < min(n.values()) and max(n.values()) <= 9472
    w = Workload(name, CASES[name], grad, "iid_normal", 0.01, tau=1, freq=4, calls=5, gemm_prec="f32", seed=3)
    sbs = SideBySide(w, gemm_prec=br.BR_GEMM_FP32, clip_norm=clip, oracle_qr="lapack")
    try:
        for c in range(6 if name == "mixed_periods" else 4):
            _, _, dg, do = sbs.step(1)
            for i, (a, b) in enumerate(zip(dg, do)):
                if b is not None:
                    assert rel_l2(a, b) <= TOL, (c, i, rel_l2(a, b))
    finally:
        sbs.close()


@pytest.mark.parametrize("m,n", [(3301, 3107), (3107, 3301)])
def test_tiles_of_128(m, n):
    """One layer whose plain launches have more than 9472 tiles of 32 x 32 (and whose paired launch takes 64 x 64 tiles
    whatever their number), rotated on its smaller side with a given orthogonal basis; result, factor and state."""
    import numpy as np
    import torch
    import paper_2602_03515_b200 as br
    from tests.parity_util import SideBySide, rel_l2
    layers = _layers([(m, n)], [GEOM_UNI], [SRC_SECOND])
    assert min(launches(layers).values()) > 9472
    w = Workload("tiles128", layers, "f32", "iid_normal", 0.01, tau=1, freq=10 ** 6, calls=3, gemm_prec="f32", seed=3)
    sbs = SideBySide(w, gemm_prec=br.BR_GEMM_FP32, oracle_qr="lapack")
    try:
        lay = sbs.oracle.layers[0]
        k = min(m, n)
        Q = np.linalg.qr(np.random.default_rng(1).standard_normal((k, k)))[0].astype(np.float32)
        setattr(lay, "U" if m <= n else "V", Q.astype(np.float64))
        sbs.opt.set_state(0, br.BR_BUF_U if m <= n else br.BR_BUF_V, torch.from_numpy(Q))
        for _ in range(3):
            _, _, dg, do = sbs.step(1)
            if do[0] is not None:
                assert rel_l2(dg[0], do[0]) <= TOL, rel_l2(dg[0], do[0])
        assert rel_l2(sbs.state(0, br.BR_BUF_L if m <= n else br.BR_BUF_R), lay.L if m <= n else lay.R) <= TOL
        assert rel_l2(sbs.state(0, br.BR_BUF_V2), lay.V2) <= TOL
    finally:
        sbs.close()
