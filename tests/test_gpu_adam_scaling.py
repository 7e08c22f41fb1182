"""The tensor-core path scales by IEEE square root and division: with bases still the identity and weights of zero, one step leaves
-lr times the bf16 rounding of M~ / sqrt(V~ + eps), to the last bit (a quotient that is an ulp off lands on the other side of a rounding
to bf16 for one entry in a hundred thousand)."""
import numpy as np
import pytest

from workloads import LayerSpec
from workloads.configs import GEOM_BI, SRC_SECOND

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1024, 2048), (520, 1544)])
def test_scaling_is_the_ieee_quotient(m, n):
    import torch
    import paper_2602_03515_b200 as br
    torch.manual_seed(3)
    W = torch.zeros(m, n, device="cuda")
    opt = br.BasisRotation([LayerSpec("w", m, n, GEOM_BI, SRC_SECOND, 1)], [W], grad_dtype="bf16", gemm_prec=br.BR_GEMM_BF16, lr=2.0 ** -10, freq=100)
    try:
        for _ in range(3):
            W.zero_()
            opt.step([(0.1 * torch.randn(m, n, device="cuda") * torch.rand(m, 1, device="cuda") ** 4).bfloat16()], 0)
        assert opt.sync_status() >= 0
        assert torch.equal(opt.get_state(0, br.BR_BUF_U), torch.eye(m)) and torch.equal(opt.get_state(0, br.BR_BUF_V), torch.eye(n))
        M, V = (opt.get_state(0, b).numpy() for b in (br.BR_BUF_MROT, br.BR_BUF_V2))
        X = M / np.sqrt(V + np.float32(1e-8))
        assert X.dtype == np.float32 and np.abs(X).max() > 1
        want = torch.from_numpy(X).bfloat16().float() * -(2.0 ** -10)
        assert torch.equal(W.cpu(), want)
    finally:
        opt.close()
