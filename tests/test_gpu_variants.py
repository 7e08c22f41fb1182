"""The library's alternative forms are selected by environment variables that are read once per
process (tuning aids: the unpaired tensor-core kernel, stream launches instead of graph replay for the
refresh, no small-order lanes, the smallest order whose refresh uses the tensor cores).  Each is
exercised here in a child process that runs a few of the ordinary parity tests under that setting, so that
the forms a user can fall back to stay correct."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(env, args):
    e = dict(os.environ)
    e.update(env)
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider"] + args,
                       cwd=ROOT, env=e, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


def test_unpaired_tensor_core_kernel():
    _run({"BR_TC_PAIR": "0"}, ["tests/test_gpu_gemm_tc.py",
                               "tests/test_gpu_full_size.py::test_c2_full_size_block_teacher_forced_bases"])


def test_refresh_without_graphs_and_small_lanes():
    _run({"BR_REFRESH_GRAPHS": "0", "BR_REFRESH_SMALL_LANES": "0", "BR_REFRESH_LANES": "1"},
         ["tests/test_gpu_full_size.py::test_refresh_order_1024_against_oracle_power",
          "tests/test_gpu_full_size.py::test_refresh_tensor_core_projections",
          "tests/test_gpu_parity_fp32.py::test_numerically_rank_deficient_refresh_is_completed_in_the_same_call",
          "tests/test_gpu_parity_bf16.py", "-k", "not checkpoint"])


def test_refresh_without_tensor_cores():
    """A raised line keeps the tensor cores out of the refresh and leaves the form of the factorisation alone."""
    _run({"BR_QR_TC_MIN_ORDER": str(1 << 30)}, ["tests/test_gpu_orth_cluster.py", "-k", "form_by_order or 1599 or 2049"])


def test_refresh_with_tensor_cores_from_order_1024():
    _run({"BR_QR_TC_MIN_ORDER": "1024"}, ["tests/test_gpu_full_size.py::test_refresh_order_1024_against_oracle_power"])


def test_steps_without_the_side_stream():
    """BR_RING_SIDE_STREAM=0 keeps a step on the handle's stream: ring copies, and small matrices beside larger ones.  The fault
    injection counts the CUDA calls of a step: none of them records an event or waits for one."""
    _run({"BR_RING_SIDE_STREAM": "0"}, ["tests/test_gpu_parity_bf16.py", "-k", "not checkpoint"])
    code = """if True:
        import torch
        import paper_2602_03515_b200 as br
        from workloads import LayerSpec
        errors = []
        for prec, dt, shapes in ((br.BR_GEMM_FP32, torch.float32, [(64, 32), (200, 130)]), (br.BR_GEMM_BF16, torch.bfloat16, [(128, 136)])):
            specs = [LayerSpec("w%d" % i, m, n, br.BR_GEOM_BILATERAL, br.BR_SRC_SECOND, 1) for i, (m, n) in enumerate(shapes)]
            for countdown in range(60):
                opt = br.BasisRotation(specs, [torch.zeros(m, n, device="cuda") for m, n in shapes], gemm_prec=prec, freq=100,
                                       grad_dtype="f32" if dt == torch.float32 else "bf16")
                g = [(0.01 * torch.randn(m, n, device="cuda")).to(dt) for m, n in shapes]
                opt.step(g, 1)
                br.br_debug_inject(opt.handle, br.BR_INJECT_LAUNCH_FAILURE, countdown)
                try:
                    opt.step(g, 1)
                    break
                except br.BrError as e:
                    errors.append(str(e))
                finally:
                    br.br_debug_inject(opt.handle, br.BR_INJECT_NONE, 0)
                    opt.close()
        assert len(errors) > 8 and not any("Event" in e or "join" in e for e in errors), errors
    """
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, BR_RING_SIDE_STREAM="0"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
