"""The fused network kernels (128-row tiles of 16 samples; weight gradients over ranges of 64-row
chunks) at the edges of their tiles and ranges, against the layer-by-layer mma.sync engine.

Both engines round the same values to BF16 and accumulate in FP32 in different orders, so a sum
that lies on a rounding boundary may round differently; the bars are those the two engines meet
against the FP64 reference (outputs 1e-3 of the largest, gradients 5e-3 of each block's norm).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 15, 16, 17, 129, 2049, 2600])  # less than a tile .. two ranges of rows, one
def test_fused_kernels_agree_with_the_layer_by_layer_engine(B):
    import paper_2205_06557_gb300 as od

    rng = np.random.default_rng(B)
    x = rng.uniform(-1.0, 1.0, (B, 8, 7))
    mask = (rng.uniform(size=(B, 8)) < 0.5).astype(np.float64)
    mask[:, 0] = 1.0
    if B > 2:
        mask[2] = 0.0  # a sample without grains
    t = rng.normal(size=(B, 8, 4))
    s = od.Surrogate(max_batch=B, seed=B)
    out = {}
    for eng in (od.GEMM_MMA_SYNC, od.GEMM_TCGEN05):
        s.set_gemm(eng)
        out[eng] = (s.forward(x, mask), *s.gradients(x, mask, t))
    s.close()
    (y0, l0, g0), (y1, l1, g1) = out[od.GEMM_MMA_SYNC], out[od.GEMM_TCGEN05]
    assert np.abs(y1 - y0).max() <= 1e-3 * np.abs(y0).max()
    assert abs(l1 - l0) <= 1e-4 * abs(l0)
    off = 0
    for o, i in od.Surrogate.SHAPES:
        for n in (o * i, o):
            a, b = g1[off: off + n].astype(np.float64), g0[off: off + n].astype(np.float64)
            off += n
            assert np.linalg.norm(a - b) <= 5e-3 * np.linalg.norm(b), (o, i, n)


def _batch(B, seed):
    rng = np.random.default_rng(seed)
    mask = (rng.uniform(size=(B, 8)) < 0.5).astype(np.float32)
    mask[:, 0] = 1.0
    return (rng.uniform(-1.0, 1.0, (B, 8, 7)).astype(np.float32), mask, rng.normal(size=(B, 8, 4)).astype(np.float32))


@pytest.mark.parametrize("max_batch", [1601, 2048, 4096])
def test_smaller_batches_of_a_large_network(max_batch):
    """Batches well below the network's largest (a training minibatch beside a held-out set) need more
    partial gradients than a full one: the same bits as in a network made for the batch."""
    import paper_2205_06557_gb300 as od

    big = od.Surrogate(max_batch=max_batch, seed=3)
    for B in (1, 16, 17, 25, 128, 1600, min(max_batch, 2048), max_batch, 128):
        args = _batch(B, B)
        one = od.Surrogate(max_batch=B, seed=3)
        (l0, g0), (l1, g1) = one.gradients(*args), big.gradients(*args)
        assert l0 == l1 and np.array_equal(g0, g1), B
        one.close()
    big.close()


def test_train_step_without_a_loss_has_read_its_inputs():
    """The caller's arrays are its own again when the call returns, page-locked ones too: they are
    overwritten at once, while the stream is still busy with work queued before the call."""
    import torch

    import paper_2205_06557_gb300 as od

    B = 512
    host = [torch.from_numpy(v).pin_memory() for v in _batch(B, 5)]
    stream = torch.cuda.Stream()
    params = []
    for overwrite in (False, True):
        net = od.Surrogate(max_batch=B, seed=1, stream=stream.cuda_stream)
        arr = [h.clone().pin_memory() for h in host]
        with torch.cuda.stream(stream):
            torch.cuda._sleep(20_000_000)  # ~10 ms
        vp = od.ctypes.c_void_p
        rc = od.lib().od_sur_train_step(net.h, *(vp(t.data_ptr()) for t in arr), B, od.ctypes.c_float(1e-3), None)
        if overwrite:
            for t in arr:
                t.fill_(0.25)
        assert rc == 0
        params.append(net.get_params())
        net.close()
    assert np.array_equal(params[0], params[1])
