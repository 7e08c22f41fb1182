"""The grouped launches of the fp32 path over several layers at once: tiles of 32, 64 and 128 (chosen by the work of
the launch), ragged edges, one-sided layers, bf16 and clipped gradients (materialised in fp32), more layers than one
launch takes, layers of a chunk that refresh while others do not -- against the float64 oracle, with the tolerance
of the other fp32 parity tests."""
import pytest

from workloads import LayerSpec, Workload
from workloads.configs import GEOM_BI, GEOM_UNI, SRC_FIRST, SRC_SECOND

pytestmark = pytest.mark.gpu
TOL = 1e-4          # relative Frobenius error of an update: fp32 chains of at most 1e3 terms through five products


def _layers(shapes, geoms, srcs, tau=1, freqs=(0,)):
    return [LayerSpec("W%d" % i, m, n, geoms[i % len(geoms)], srcs[i % len(srcs)], tau, freqs[i % len(freqs)])
            for i, (m, n) in enumerate(shapes)]


CASES = {
    "tiles32_ragged": _layers([(131, 33), (33, 140), (200, 129)], [GEOM_BI, GEOM_UNI], [SRC_SECOND]),
    "tiles64": _layers([(1100, 260), (260, 1301)], [GEOM_UNI], [SRC_SECOND]),
    "tiles128": _layers([(1400, 1300), (130, 3300)], [GEOM_UNI], [SRC_SECOND]),
    "many": _layers([(130 + i, 20 + i) for i in range(35)], [GEOM_UNI, GEOM_BI], [SRC_SECOND]),
    "mixed_periods": _layers([(140, 139), (150, 40), (40, 150)], [GEOM_BI, GEOM_UNI], [SRC_SECOND, SRC_FIRST], freqs=(2, 3, 5)),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("grad,clip", [("f32", 0.0), ("bf16", 0.5)])
def test_group(name, grad, clip):
    import paper_2602_03515_b200 as br
    from tests.parity_util import SideBySide, rel_l2
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
