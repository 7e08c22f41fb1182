"""The one-launch update of small matrices (fp32, both dimensions at most 128) against the float64 oracle: both forms of
its kernel (a dot product per thread for a few hundred entries, tiles otherwise), the tiled form on a cluster of one
CTA (no dimension of 32 or more) and of four, one and both rotated sides, sizes at the edges of the rule between the
forms, and more matrices than one launch takes.  Both sides are given the same random orthogonal bases (a refresh of
the elongated shapes would complete a rank-deficient product, which says little about the arithmetic of a step)."""
import numpy as np
import pytest

from workloads import LayerSpec, Workload
from workloads.configs import GEOM_BI, GEOM_UNI, SRC_FIRST, SRC_SECOND

pytestmark = pytest.mark.gpu
TOL = 1e-4          # relative Frobenius error of an update: as for the other fp32 parity tests

SINGLE = [(1, 1), (1, 5), (8, 8), (16, 8), (17, 30), (22, 22), (23, 22), (24, 24), (30, 31), (31, 31), (32, 4), (31, 33),
          (48, 20), (64, 8), (128, 2), (2, 128), (128, 4), (127, 3), (100, 9), (40, 25), (32, 32), (128, 7)]
GROUPS = {
    "tiny": [(5 + i % 13, 4 + i % 9) for i in range(30)],
    "below32": [(24 + i % 8, 31 - i % 8) for i in range(26)],
    "mixed": [(64, 32), (7, 9), (30, 30), (3, 128), (100, 40), (16, 16), (33, 77)] * 7,
}


def _run(shapes, geoms, srcs, grad, clip):
    import torch
    import paper_2602_03515_b200 as br
    from tests.parity_util import SideBySide, rel_l2
    layers = [LayerSpec("W%d" % i, m, n, geoms[i % len(geoms)], srcs[i % len(srcs)], 1) for i, (m, n) in enumerate(shapes)]
    w = Workload("small", layers, grad, "iid_normal", 0.01, tau=1, freq=10 ** 6, calls=5, gemm_prec="f32", seed=5)
    sbs = SideBySide(w, gemm_prec=br.BR_GEMM_FP32, clip_norm=clip, oracle_qr="lapack")
    rng = np.random.default_rng(7)
    try:
        for i, lay in enumerate(sbs.oracle.layers):
            for side, which in (("U", br.BR_BUF_U), ("V", br.BR_BUF_V)):
                if getattr(lay, side) is not None:
                    Q = np.linalg.qr(rng.standard_normal(getattr(lay, side).shape))[0].astype(np.float32)
                    setattr(lay, side, Q.astype(np.float64))
                    sbs.opt.set_state(i, which, torch.from_numpy(Q))
        for c in range(5):
            _, _, dg, do = sbs.step(1)
            for i, (a, b) in enumerate(zip(dg, do)):
                if b is not None:
                    assert rel_l2(a, b) <= TOL, (c, i, shapes[i], rel_l2(a, b))
        for i, lay in enumerate(sbs.oracle.layers):
            for which, ref in ((br.BR_BUF_M, lay.M), (br.BR_BUF_V2, lay.V2), (br.BR_BUF_L, lay.L), (br.BR_BUF_R, lay.R)):
                if ref is not None:
                    assert rel_l2(sbs.state(i, which), ref) <= TOL, (i, shapes[i], which)
    finally:
        sbs.close()


@pytest.mark.parametrize("m,n", SINGLE)
@pytest.mark.parametrize("geom,src", [(GEOM_BI, SRC_SECOND), (GEOM_UNI, SRC_SECOND), (GEOM_UNI, SRC_FIRST)])
def test_one_matrix(m, n, geom, src):
    _run([(m, n)], [geom], [src], "f32", 0.0)


@pytest.mark.parametrize("name", sorted(GROUPS))
@pytest.mark.parametrize("grad,clip", [("f32", 0.0), ("bf16", 0.5)])
def test_more_than_one_launch(name, grad, clip):
    _run(GROUPS[name], [GEOM_BI, GEOM_UNI], [SRC_SECOND, SRC_FIRST, SRC_SECOND], grad, clip)
