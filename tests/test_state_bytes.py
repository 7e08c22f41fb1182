"""How much device memory a handle asks for (br_state_bytes, host only): state plus scratch of the refresh lanes."""
import pytest

import paper_2602_03515_b200 as br
from workloads.configs import GEOM_BI, GEOM_UNI, SRC_FIRST, SRC_SECOND


@pytest.fixture(scope="module", autouse=True)
def library():
    import __graft_entry__ as ge
    ge.build()


def total_bytes(shapes, geom, src, prec, tau=4):
    grad = br.BR_BF16 if prec == br.BR_GEMM_BF16 else br.BR_F32
    descs = [br.BrLayerDesc(m=m, n=n, geom=geom, src=src, grad_dtype=grad, tau_max=tau, freq=0, reserved=0, weight=4096) for m, n in shapes]
    hp = br.BrHparams(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, beta_factor=-1.0, freq=10, power_iters=1,
                      accum=0, gemm_prec=prec, flags=0, clip_norm=0.0, scratch_limit_bytes=0)
    return br.br_state_bytes(descs, hp)[0]


def block(d, ffn, n=1):
    return [(d, 3 * d), (d, d), (d, ffn), (ffn, d)] * n


@pytest.mark.parametrize("k", [64, 1000, 1599])
def test_a_lane_of_one_launch_orders(k):
    """One one-sided k x k layer: state M, V~, U, L, scratch of the step 4 k^2 floats, and one lane with the product, its
    copy (k^2 doubles each) and the factorisation's work (coefficients k^2 / 4, column norms 2 x 16 k, diagonal k)."""
    want = 4 * 4 * k * k + 4 * 4 * k * k + 8 * (2 * k * k + k * k / 4 + 33 * k)
    assert total_bytes([(k, k)], GEOM_UNI, SRC_SECOND, br.BR_GEMM_FP32, tau=0) <= want + 16 * 1024 + 8 * k


@pytest.mark.parametrize("emb,d,ffn", [(32000, 1536, 6144), (50257, 768, 3072)])
def test_first_source_buffers_do_not_grow_with_the_largest_matrix(emb, d, ffn):
    """The half product of an S = 1st refresh has at most 128 MiB in each of at most eight lanes."""
    blk = total_bytes(block(d, ffn), GEOM_UNI, SRC_FIRST, br.BR_GEMM_BF16)
    both = total_bytes([(emb, d)] + block(d, ffn), GEOM_UNI, SRC_FIRST, br.BR_GEMM_BF16)
    tc = emb % 8 == 0
    # the layer itself: M, V~ (and the momentum of the original space), ring of four bf16 slots, basis and its bf16 pair; on
    # the fp32 path its step's scratch of 4 m n floats, on the tensor-core path the operands of its chunk, 11 bytes an entry
    layer = emb * d * (8 + (4 + 11 if tc else 16) + 4 * 2) + d * d * 8
    lane = 8 * (2 * d * d + d * d / 4 + 33 * d)
    assert both - blk <= layer + 8 * (128 << 20) + 2 * lane
