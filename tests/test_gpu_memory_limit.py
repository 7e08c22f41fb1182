"""A handle whose allocator refuses the usual layout gets the one with three full-size refresh lanes, which asks for no
more than a third of the lanes' memory; a set for which that is not smaller is refused at once."""
import pytest

from workloads import LayerSpec
from workloads.configs import GEOM_BI, GEOM_UNI, SRC_SECOND

pytestmark = pytest.mark.gpu

SHAPES = [(384, 350), (329, 384), (200, 210), (184, 190), (297, 300)]


class _Limited:
    """A device allocator that refuses requests above `limit` bytes."""

    def __init__(self, limit):
        import torch
        from paper_2602_03515_b200 import binding as B
        self.asked, self.blocks = [], {}

        def alloc(nbytes, _ctx):
            self.asked.append(int(nbytes))
            if nbytes > limit:
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.blocks[t.data_ptr()] = t
            return t.data_ptr()

        self.cb = (B._ALLOC_FN(alloc), B._FREE_FN(lambda ptr, _ctx: self.blocks.pop(ptr, None)))
        self.struct = B.BrAllocator(self.cb[0], self.cb[1], None)


def _create(br, weights, limit, geom, shapes=SHAPES, dtype=0):
    specs = [LayerSpec("w", m, n, geom, SRC_SECOND, 1) for m, n in shapes[:len(weights)]]
    descs = [br.BrLayerDesc(m=s.m, n=s.n, geom=s.geom, src=s.src, grad_dtype=dtype, tau_max=1, freq=0, reserved=0,
                            weight=w.data_ptr()) for s, w in zip(specs, weights)]
    hp = br.BrHparams(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, beta_factor=-1.0, freq=3, power_iters=1,
                      accum=0, gemm_prec=br.BR_GEMM_BF16 if dtype else br.BR_GEMM_FP32, flags=0, clip_norm=0.0, scratch_limit_bytes=0)
    a = _Limited(limit)
    try:
        return a, br.br_state_bytes(descs, hp)[0], br.br_create(descs, hp, 0, 0, a.struct)
    except br.BrError as e:
        return a, br.br_state_bytes(descs, hp)[0], e


def test_smaller_layout_after_a_refusal():
    import torch
    import paper_2602_03515_b200 as br
    torch.manual_seed(1)
    W0 = [0.02 * torch.randn(m, n, device="cuda") for m, n in SHAPES]
    G = [[0.01 * torch.randn(m, n, device="cuda") for m, n in SHAPES] for _ in range(3)]
    torch.cuda.synchronize()
    results = []
    usual = None
    for limited in (False, True):
        W = [w.clone() for w in W0]
        torch.cuda.synchronize()
        a, usual, h = _create(br, W, usual - 1 if limited else 1 << 60, GEOM_BI)
        assert not isinstance(h, Exception), h
        try:
            assert len(a.asked) == (2 if limited else 1) and a.asked[0] >= usual
            if limited:
                assert a.asked[1] < 0.7 * usual
            for c in range(8):
                br.br_step(h, [g.data_ptr() for g in G[c % 3]], 1)
            assert br.br_sync_status(h) >= 0
            results.append(W)
        finally:
            br.br_destroy(h)
        assert not a.blocks
    # (the layers' fp32 products run in other groups, and with them in other tiles: the tolerance of the fp32 parity tests)
    for x, y, w in zip(*results, W0):
        assert torch.linalg.norm(x - y) <= 1e-4 * torch.linalg.norm(y - w)


def test_no_second_request_where_nothing_is_smaller():
    import torch
    import paper_2602_03515_b200 as br
    W = [torch.zeros(m, n, device="cuda") for m, n in SHAPES[:1]]
    a, usual, e = _create(br, W, 0, GEOM_UNI)
    assert isinstance(e, br.BrError) and e.status == br.BR_ERR_OOM
    assert len(a.asked) == 1 and not a.blocks
    a, usual, e = _create(br, W, 1 << 60, GEOM_UNI)
    br.br_destroy(e)


@pytest.mark.parametrize("d,blocks,limit", [(456, 3, 807 << 20), (528, 2, 1091 << 20)])
def test_smaller_layout_beside_lanes(d, blocks, limit):
    """Orders on both sides of 1600: lanes for the ones above, a pool for the others.  The smaller layout fits where three lanes that
    hold every order do (791 and 1077 MiB)."""
    import torch
    import paper_2602_03515_b200 as br
    shapes = [(d, 3 * d), (d, d), (d, 4 * d), (4 * d, d)] * blocks
    W = [0.02 * torch.randn(m, n, device="cuda") for m, n in shapes]
    G = [(0.01 * torch.randn(m, n, device="cuda")).bfloat16() for m, n in shapes]
    before = [w.clone() for w in W]
    torch.cuda.synchronize()
    a, usual, h = _create(br, W, limit, GEOM_BI, shapes, br.BR_BF16)
    assert not isinstance(h, Exception), (h, a.asked)
    try:
        assert len(a.asked) == 2 and a.asked[1] <= limit < a.asked[0]
        for _ in range(7):
            br.br_step(h, [g.data_ptr() for g in G], 1)
        assert br.br_sync_status(h) >= 0 and all(torch.isfinite(w).all() and not torch.equal(w, b) for w, b in zip(W, before))
    finally:
        br.br_destroy(h)
