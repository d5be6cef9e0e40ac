"""A bounded wait of the network's tensor-core forward that runs out (test hook: a barrier that also waits for
bytes that no copy brings) leaves NaN and is reported once, by the next call."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TEST_TIMEOUT = -0x7FFFFFFF


@pytest.fixture(scope="module")
def ue():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    return ue


@pytest.mark.parametrize("call", ["forward", "backward", "adam", "argmax", "loss"])
def test_a_forward_that_ran_out_of_time_is_reported(ue, call):
    import torch
    from paper_1812_01448_gb300 import _native as N
    g = torch.Generator(device="cuda").manual_seed(2)
    n, k = 40_001, N.UE_MLP_PARAMS
    P = torch.randn(k, device="cuda", generator=g) * 0.2
    X = torch.randn(n, 12, device="cuda", generator=g)
    base = torch.zeros(n, device="cuda")
    z, ref = torch.zeros(n, device="cuda"), torch.empty(n, device="cuda")
    ue.mlp_forward(P, X, ref)
    p = lambda t: C.c_void_p(t.data_ptr())
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    N.check(N.lib().ue_mlp_forward(p(P), p(X), n, TEST_TIMEOUT, p(z), s), "forward")
    torch.cuda.synchronize()
    bad = torch.isnan(z)
    assert 0 < int(bad.sum()) < n and torch.equal(z[~bad], ref[~bad])
    off = torch.tensor([0, n], device="cuda")
    best, arg = torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    rows, dz, work, grad = arg.clone(), best.clone(), torch.empty(k, device="cuda"), torch.zeros(k, device="cuda")
    run = {"forward": lambda: ue.mlp_forward(P, X, z), "backward": lambda: ue.mlp_backward(P, X, rows, dz, grad, work),
           "adam": lambda: ue.adam(P.clone(), grad, grad.clone(), grad.clone(), 1),
           "argmax": lambda: ue.seg_argmax(z, base, off, best, arg),
           "loss": lambda: ue.rho_loss(best, best.clone(), dz, work[:1])}[call]
    with pytest.raises(ue.UEError) as e:
        run()
    assert e.value.code == -8
    run()                                  # reported once
    ue.mlp_forward(P, X, z)
    ue.seg_argmax(z, base, off, best, arg)
    torch.cuda.synchronize()
    assert torch.equal(z, ref) and int(arg) == int(torch.argmax(ref)) and np.isfinite(float(best))


def test_the_first_forward_may_be_captured(ue):
    """The word that reports a failure is made on the first use, also inside a capture."""
    import subprocess
    import sys
    code = """
import torch, paper_1812_01448_gb300 as ue
P, X = torch.randn(5057, device="cuda") * 0.2, torch.randn(40000, 12, device="cuda")
z = torch.zeros(40000, device="cuda")
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    ue.mlp_forward(P, X, z)
g.replay()
a = z.clone()
ue.mlp_forward(P, X, z)
torch.cuda.synchronize()
assert torch.equal(a, z) and float(z.abs().sum()) > 0
"""
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)
