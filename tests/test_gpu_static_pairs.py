"""od_pair_accel_static at the edges of its tiles (256 targets), source chunks and of its two kernel
forms (up to 2,048 padded ions, and above), against an FP64 sum of the same positions: per ion
within 1e-5 of the sum of the term magnitudes (the bar of the injected-state force tests), and
the same bits from a repeated call."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 255, 257, 2048, 2049, 10007, 32768])
def test_static_accelerations_match_fp64(n):
    import paper_2205_06557_gb300 as od
    from paper_2205_06557_gb300 import workloads as W

    lam, k = 1.66e-3, 3.5e-3
    x, _, _ = W.random_ions(n, 2e-4, 4e-4, seed=n)
    xd = torch.from_numpy(x).cuda()
    out = []
    for _ in range(2):
        a = torch.full((n, 3), float("nan"), dtype=torch.float32, device="cuda")
        od.od_pair_accel_static(xd.data_ptr(), n, lam, k, a.data_ptr())
        torch.cuda.synchronize()
        out.append(a)
    assert torch.equal(out[0], out[1])
    ref = torch.zeros_like(xd)
    mag = torch.zeros(n, dtype=torch.float64, device="cuda")
    for i in range(0, n, 512):
        d = xd[i: i + 512, None, :] - xd[None, :, :]
        r = d.square().sum(2).sqrt()
        c = k * (1 + r / lam) * torch.exp(-r / lam) / r ** 3
        c[r == 0] = 0.0
        ref[i: i + 512] = (c[..., None] * d).sum(1)
        mag[i: i + 512] = (c * r).sum(1)
    err = (out[0].double() - ref).norm(dim=1)
    assert bool((err <= 1e-5 * mag).all()), float((err / mag).max())


@pytest.mark.parametrize("n", [300, 3001])  # both kernel forms
def test_captured_call_replays(n):
    """A captured call gives an uncaptured call's bits on every replay, with the positions of that
    replay: many close pairs, the lists of one replay must not reach the next."""
    import paper_2205_06557_gb300 as od
    from paper_2205_06557_gb300 import workloads as W

    lam, k = 1.66e-3, 3.5e-3
    R = 2e-5 * (n / 300) ** (1 / 3)  # a few neighbours within the correction distance
    xs = [torch.from_numpy(W.random_ions(n, R, 2 * R, seed=s)[0]).cuda() for s in (1, 2)]
    x = xs[0].clone()
    a = torch.empty((n, 3), dtype=torch.float32, device="cuda")

    def call():
        od.od_pair_accel_static(x.data_ptr(), n, lam, k, a.data_ptr(), torch.cuda.current_stream().cuda_stream)

    ref = []
    for s in xs:
        x.copy_(s)
        call()
        torch.cuda.synchronize()
        ref.append(a.clone())
    assert not torch.equal(ref[0], ref[1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    for r in (0, 0, 1, 0):
        x.copy_(xs[r])
        a.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, ref[r])
    call()  # and an uncaptured call after them
    torch.cuda.synchronize()
    assert torch.equal(a, ref[0])
