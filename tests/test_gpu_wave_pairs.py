"""The ordered kernel's block sums made from unordered pairs (variant k_forces<128,2>, 7,681 to 32,768
padded ions) at the edges of that range, with ragged last tiles and other plans, against an FP64 sum of
the same positions: per ion within 1e-5 of the sum of the term magnitudes (the bar of the
injected-state force tests), and the same bits from a repeated evaluation."""
import math

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,upb,bps", [(7680, 8, 0), (7681, 8, 0), (10241, 8, 0), (12032, 1, 0), (12033, 64, 2), (20011, 8, 0),
                                       (20011, 1000, 1), (32768, 8, 0), (32769, 8, 0)])
def test_wave_accelerations_match_fp64(n, upb, bps):
    import paper_2205_06557_gb300 as od
    from paper_2205_06557_gb300 import workloads as W

    p = W.plasma_ar()
    R = (n / p["n_inf"] / (2 * math.pi)) ** (1 / 3)
    p.update(R=R, H=2 * R, dt=5e-10, n_ions=n, seed=1, charge_model="given", dust=[], avg_start=1, flags=od.F_NO_EOUT)
    d = oracle.Oracle(dict(p, n_ions=1)).derived()
    drift = d["q"] * d["E"] / d["m"]  # the flow field's term, along z
    lam, k = d["lam"], d["q"] ** 2 / (4 * math.pi * 8.8541878128e-12 * d["m"])
    x, v, ids = W.random_ions(n, p["R"], p["H"], seed=n)
    run = od.Run(p)
    od.od_set_force_config(run.h, 2, upb, bps)
    acc = []
    for _ in range(2):
        run.set_ions(x, v, ids, next_id=n)
        acc.append(run.get_ions()[2].copy())
    run.close()
    assert np.array_equal(acc[0], acc[1])
    xd, a = torch.from_numpy(x).cuda(), torch.from_numpy(acc[0]).cuda().double()
    for i in range(0, n, 512):
        s = xd[i: i + 512, None, :] - xd[None, :, :]
        r = s.square().sum(2).sqrt()
        c = k * (1 + r / lam) * torch.exp(-r / lam) / r ** 3
        c[r == 0] = 0.0
        ref, mag = (c[..., None] * s).sum(1), (c * r).sum(1) + drift
        ref[:, 2] += drift
        err = (a[i: i + 512] - ref).norm(dim=1)
        assert bool((err <= 1e-5 * mag).all()), float((err / mag).max())


@pytest.mark.parametrize("tiles,upb,bps", [(16, 1, 2), (16, 3, 2), (19, 1, 1), (19, 8, 1), (32, 2, 4), (38, 1, 1), (38, 5, 1),
                                           (38, 64, 1)])
@pytest.mark.parametrize("short", [0, 61])
def test_wave_block_sums_are_the_ordered_kernels(tiles, upb, bps, short):
    """Bit for bit the accelerations of the ordered kernel with 512-ion tiles, k_forces<128,4>: it adds the
    same blocks of 128 sources in the same order, and under these plans its CTAs split each target's
    sources at the same places (the CTAs per tile divide evenly, half the tile width and twice the
    CTAs for k_forces<128,2>).  Ragged last tiles, one to many chunks per CTA."""
    import paper_2205_06557_gb300 as od
    from paper_2205_06557_gb300 import workloads as W

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms * bps % tiles:
        pytest.skip("the plans split their tiles evenly on 152 SMs")
    n = 512 * tiles - short
    p = W.plasma_ar()
    R = (n / p["n_inf"] / (2 * math.pi)) ** (1 / 3)
    p.update(R=R, H=2 * R, dt=5e-10, n_ions=n, seed=1, charge_model="given", dust=[], avg_start=1, flags=od.F_NO_EOUT)
    x, v, ids = W.random_ions(n, p["R"], p["H"], seed=n)
    run = od.Run(p)
    acc = []
    for variant, b in ((2, 2 * bps), (3, bps)):
        assert od.force_variant_name(variant) == "k_forces<128,%d>" % (2 if variant == 2 else 4)
        od.od_set_force_config(run.h, variant, upb, b)
        run.set_ions(x, v, ids, next_id=n)
        acc.append(run.get_ions()[2].copy())
    run.close()
    assert np.array_equal(acc[0], acc[1])
