"""Observability and restart through the C ABI: checkpoints continue bit for bit, the
density map equals a host binning of the same positions, ion dumps hold the exact state."""
import math

import numpy as np
import pytest

import paper_2205_06557_gb300 as od
from paper_2205_06557_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2205_06557_gb300 import build

    build.build()
    od.lib()


def _medium():
    """~40,000 ions: above the size where the untuned run uses the symmetric kernel"""
    p = W.tiny()
    p["R"] *= 2.72
    p["H"] *= 2.72
    p["n_ions"] = 0
    return p


@pytest.mark.parametrize("make", [W.tiny, _medium])
def test_checkpoint_continues_bit_for_bit(make, tmp_path):
    p = make()
    p["avg_start"] = 5
    a = od.Run(p)
    a.step(12)
    path = str(tmp_path / "run.ckpt")
    a.save(path)
    a.step(13)
    b = od.Run.load(path)
    assert b.D == a.D and b.N == a.N
    assert od.od_get_force_config(b.h)[:3] == od.od_get_force_config(a.h)[:3]
    b.step(13)
    ra, ea = a.series(1, 25)
    rb, eb = b.series(1, 25)
    assert np.array_equal(ea, eb) and np.array_equal(ra, rb)
    xa, va, aa, ia = a.get_ions()
    xb, vb, ab, ib = b.get_ions()
    assert np.array_equal(ia, ib) and np.array_equal(xa, xb) and np.array_equal(va, vb) and np.array_equal(aa, ab)
    for fa, fb in zip(a.dust_state() + a.dust_terms(), b.dust_state() + b.dust_terms()):
        assert np.array_equal(fa, fb)
    assert np.array_equal(a.counters(), b.counters())
    a.close()
    b.close()


def _bin(x, R, H, nr, nz):
    """host binning with the library's stated FP64 formula (numpy does not contract)"""
    r = np.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1])
    ir = np.clip(np.floor(r * (nr / R)).astype(np.int64), 0, nr - 1)
    iz = np.clip(np.floor((x[:, 2] + 0.5 * H) * (nz / H)).astype(np.int64), 0, nz - 1)
    out = np.zeros((nz, nr), dtype=np.uint64)
    np.add.at(out, (iz, ir), 1)
    return out


@pytest.mark.parametrize("nr,nz", [(16, 32), (128, 128)])  # shared-memory and global-atomic paths
def test_density_map_equals_host_binning(nr, nz):
    p = W.tiny()
    run = od.Run(p)
    run.step(3)
    od.od_density_enable(run.h, nr, nz)
    ref = np.zeros((nz, nr), dtype=np.uint64)
    for _ in range(15):
        run.step(1)
        ref += _bin(run.get_ions()[0], p["R"], p["H"], nr, nz)
    counts, dens, n = od.od_density_read(run.h, nr, nz)
    assert n == 15 and np.array_equal(counts, ref)
    assert int(counts.sum()) == 15 * run.N
    # density x annulus volume, summed, gives back the ion count per step
    r = np.linspace(0, p["R"], nr + 1)
    vol = math.pi * (r[1:] ** 2 - r[:-1] ** 2)[None, :] * (p["H"] / nz)
    assert np.isclose((dens * vol).sum(), run.N, rtol=1e-12)
    # mean density is the ion count over the cylinder volume
    assert np.isclose((dens * vol).sum() / (math.pi * p["R"] ** 2 * p["H"]), run.N / (math.pi * p["R"] ** 2 * p["H"]))
    od.od_density_enable(run.h, 0, 0)
    run.step(2)
    with pytest.raises(od.OdError):
        od.od_density_read(run.h, nr, nz)
    run.close()


def test_bad_density_map_sizes_are_rejected():
    run = od.Run(W.tiny())
    for nr, nz in [(-1, 4), (5000, 4), (4096, 4096), (0, 3)]:
        with pytest.raises(od.OdError) as ei:
            od.od_density_enable(run.h, nr, nz)
        assert ei.value.code == -1
    run.close()


def test_ion_dumps_hold_the_exact_state(tmp_path):
    run = od.Run(W.tiny())
    run.step(4)
    x, v, _, ids = run.get_ions()
    xyz = str(tmp_path / "ions.xyz")
    csv = str(tmp_path / "ions.csv")
    run.write_ions(xyz, od.DUMP_XYZ)
    run.write_ions(csv, od.DUMP_CSV)
    lines = open(xyz).read().splitlines()
    assert int(lines[0]) == run.N and "step=4" in lines[1]
    body = np.array([ln.split()[1:] for ln in lines[2:]], dtype=np.float64)
    assert np.array_equal(body[:, :3], x) and np.array_equal(body[:, 3:6], v)
    assert np.array_equal(np.array([ln.split()[7] for ln in lines[2:]], dtype=np.uint64), ids)
    c = np.loadtxt(csv, delimiter=",", skiprows=1, dtype=np.float64)
    assert np.array_equal(c[:, 1:4], x) and np.array_equal(c[:, 4:7], v)
    assert np.array_equal(np.loadtxt(csv, delimiter=",", skiprows=1, usecols=0, dtype=np.uint64), ids)
    run.close()


def test_kernel_times_span_more_steps_than_the_event_ring():
    """per-kernel profiling records events for every step and reads them 64 steps at a
    time: a call of 70 steps and one of 5 count 75 launches of each stage, and the
    profiled (directly launched) steps give the same bits as graph-replayed ones (75 steps
    in one call: four 16-step graphs and eleven one-step graphs), state and records"""
    p = W.tiny(steps=200)
    prof, ref = od.Run(p), od.Run(p)
    od.od_set_profiling(prof.h, 1)
    prof.step(70)
    prof.step(5)
    ms, n = od.od_kernel_times(prof.h)
    assert n.tolist() == [75] * 4 and (ms > 0).all()
    od.od_set_profiling(prof.h, 0)
    ref.step(75)
    for a, b in zip(prof.get_ions(), ref.get_ions()):
        assert np.array_equal(a, b)
    for a, b in zip(prof.series(1, 75), ref.series(1, 75)):
        assert np.array_equal(a, b)
    prof.close()
    ref.close()


def test_step_graph_lengths_give_the_same_bits():
    """od_step replays 16-step graphs while 16 or more steps remain and one-step graphs for
    the rest: 40 steps as one call, as 16 + 1 + 23, and one at a time end in the same state
    and records"""
    p = W.tiny(steps=200)
    runs = [od.Run(p) for _ in range(3)]
    runs[0].step(40)
    for k in (16, 1, 23):
        runs[1].step(k)
    for _ in range(40):
        runs[2].step(1)
    ref_state, ref_series = runs[0].get_ions(), runs[0].series(1, 40)
    for r in runs[1:]:
        for a, b in zip(r.get_ions(), ref_state):
            assert np.array_equal(a, b)
        for a, b in zip(r.series(1, 40), ref_series):
            assert np.array_equal(a, b)
    for r in runs:
        r.close()


def test_host_arrays_used_in_place_lie_in_one_page_locked_range():
    """an array whose two ends are page-locked by two registrations, with pageable memory between, is
    not handed to a kernel; pieces of one registration or allocation are (host side only)"""
    import mmap

    import torch

    page, rt = 65536, torch.cuda.cudart()
    buf = mmap.mmap(-1, 4 * page)
    raw = np.frombuffer(buf, dtype=np.uint8)
    raw[:] = 1
    p0 = -(-raw.ctypes.data // page) * page  # two whole pages with one between
    assert not od.od_selftest_host_direct(p0, 3 * page)
    for p in (p0, p0 + 2 * page):
        assert int(rt.cudaHostRegister(p, page, 0)) == 0
    try:
        for p in (p0, p0 + 2 * page):
            assert od.od_selftest_host_direct(p, page)
            assert od.od_selftest_host_direct(p + 8, page - 8)
            assert not od.od_selftest_host_direct(p + 4, 64)
        assert not od.od_selftest_host_direct(p0, 3 * page)
        assert not od.od_selftest_host_direct(p0 + 8, 2 * page)
        assert not od.od_selftest_host_direct(p0, page + 8)
    finally:
        for p in (p0, p0 + 2 * page):
            rt.cudaHostUnregister(p)
    t = torch.zeros(5000, dtype=torch.float64, pin_memory=True)
    assert od.od_selftest_host_direct(t.data_ptr(), 40000) and od.od_selftest_host_direct(t.data_ptr() + 800, 39200)
    assert not od.od_selftest_host_direct(t.data_ptr(), 1 << 40)


def test_checkpoint_without_ions(tmp_path):
    """a state without ions stays one across a checkpoint: the reads give no ions (the plan of the
    restored run is still the creation's), and a state put in afterwards is read back whole"""
    p = W.tiny()
    a = od.Run(p)
    a.set_ions(np.zeros((0, 3)), np.zeros((0, 3)), np.zeros(0, dtype=np.uint64), next_id=7)
    assert len(a.get_ions()[0]) == 0
    path = str(tmp_path / "empty.ckpt")
    a.save(path)
    b = od.Run.load(path)
    assert all(len(t) == 0 for t in b.get_ions()) and b.counters()[14] == 0
    x, v, ids = W.random_ions(100, p["R"], p["H"], seed=3, dust=p["dust"])
    b.set_ions(x, v, ids, next_id=100)
    xb, vb, _, ib = b.get_ions()
    assert np.array_equal(xb, x) and np.array_equal(vb, v) and np.array_equal(ib, ids)
    a.close()
    b.close()


@pytest.mark.parametrize("grains", [0, 1, 3])
def test_series_of_any_length_are_parts_of_the_whole(grains):
    """ranges below and above the length from which they are copied whole, ragged ones, records or events
    alone: the parts of the whole series"""
    p = W.tiny()
    p["dust"] = [dict(x=0.0, y=0.0, z=6e-5 * (k - 1), a=1e-5, q0=-2e-15) for k in range(grains)]
    r = od.Run(p)
    r.step(300)
    rec, ev = (np.concatenate(v) for v in zip(*(r.series(s, 50) for s in range(1, 301, 50))))
    assert rec.shape[:2] == (300, grains) and ev.shape[0] == 300 and ev.any()
    for first, count in ((1, 300), (1, 256), (2, 257), (3, 129), (17, 128), (300, 1), (5, 0)):
        a, b = r.series(first, count)
        assert np.array_equal(a, rec[first - 1: first - 1 + count]) and np.array_equal(b, ev[first - 1: first - 1 + count])
    for count in (200, 290):
        a, b = np.zeros_like(rec[:count]), np.zeros_like(ev[:count])
        assert od.lib().od_series(r.h, 1, count, a.ctypes.data, None) == 0 and np.array_equal(a, rec[:count])
        assert od.lib().od_series(r.h, 1, count, None, b.ctypes.data) == 0 and np.array_equal(b, ev[:count])
    r.close()
