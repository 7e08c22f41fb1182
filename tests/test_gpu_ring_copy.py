"""Gradients into the ring: several in one launch of the library's kernel, more than a launch takes, sizes that no 16-byte piece
divides, large ones among small ones; and the launch count, which has the kernel in it."""
import pytest

from workloads import LayerSpec
from workloads.configs import GEOM_BI, GEOM_NONE, SRC_SECOND

pytestmark = pytest.mark.gpu


def _run(shapes, dtype, geom, prec, calls=3):
    import torch
    import paper_2602_03515_b200 as br
    specs = [LayerSpec("w%d" % i, m, n, geom, SRC_SECOND, 2) for i, (m, n) in enumerate(shapes)]
    ws = [torch.zeros(m, n, device="cuda") for m, n in shapes]
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    opt = br.BasisRotation(specs, ws, grad_dtype=dtype, gemm_prec=getattr(br, prec), freq=100)
    try:
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1)
        sent, launches = [], []
        for _ in range(calls):
            sent.append([(0.01 * torch.randn(m, n, device="cuda", generator=gen)).to(tdt) for m, n in shapes])
            before = opt.launch_stats()[0]
            opt.step(sent[-1], 2)
            launches.append(opt.launch_stats()[0] - before)
        assert opt.sync_status() == br.BR_OK
        for i in range(len(shapes)):                      # slot (call - 1) mod 2 holds call's gradient
            ring = opt.get_state(i, br.BR_BUF_RING).cpu().reshape(2, *shapes[i])
            for call in (calls - 1, calls):
                assert torch.equal(ring[(call - 1) % 2], sent[call - 1][i].cpu()), (i, call)
        return launches
    finally:
        opt.close()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_many_and_ragged(dtype):
    """Sizes around the 16-byte pieces (bf16: 2 to 34 bytes), seventy-one gradients (two launches), one of more than 4 MiB."""
    shapes = [(1, k) for k in (1, 2, 3, 7, 8, 9, 15, 16, 17)] + [(37, 53), (5, 1999)] + [(13, 17)] * 59 + [(1100, 1999)]
    launches = _run(shapes, dtype, GEOM_NONE, "BR_GEMM_FP32")
    assert launches == [2, 2, 2 + len(shapes)]            # copies; the third call updates every matrix too


def test_one_gradient_is_a_plain_copy():
    assert _run([(300, 100)], "f32", GEOM_NONE, "BR_GEMM_FP32") == [0, 0, 1]


def test_beside_the_contractions():
    """Tensor-core layers: 66 small gradients, two launches, by themselves in the first calls and on the side stream of an update, where
    one of 4 MiB or more is copied by itself."""
    launches = _run([(16, 24)] * 66 + [(1536, 1400)], "bf16", GEOM_BI, "BR_GEMM_BF16")
    assert launches[:2] == [2, 2] and launches[2] > 2
