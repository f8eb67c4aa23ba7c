"""What the autotuner times for the half apply's layouts is a whole S apply: the time it reports for the layout it
chose is that of the reduced operator, not of one half alone (whose order differs from that of the pair)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_reported_time_is_the_operators():
    import paper_2205_09104_gb300 as cg
    dims, nv = (8, 8, 8, 8), 16
    V, n = int(np.prod(dims)), 2 * nv
    g = torch.Generator(device="cuda").manual_seed(5)
    f = 0.05 * torch.randn(V, 4, n, n, dtype=torch.complex128, device="cuda", generator=g)
    s = 2.5 * torch.eye(n, dtype=torch.complex128, device="cuda").repeat(V, 1, 1)
    dev = cg.CoarseOp(s, f, dims, nv, precisions=(cg.PREC_FP32,), assume_gamma5=True)
    x = torch.randn(V * n // 2, dtype=torch.complex64, device="cuda", generator=g)
    key = f"eo/p1/n{n}/v{V.bit_length() - 1}"
    cg.autotune_set(key, -1)
    dev.schur(x, precision=1)
    line = [r for r in cg.autotune_report().splitlines() if r.startswith(key)][0]
    reported = float(line.split("|")[0].split()[-1])
    times = []
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(20):
            dev.schur(x, precision=1)
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1) * 1e3 / 20)
    assert 0.75 * min(times) <= reported <= 1.5 * min(times), (line, times)
    cg.autotune_set(key, -1)
    dev.close()
