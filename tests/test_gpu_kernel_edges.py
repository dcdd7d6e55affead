"""Edges of the step and adjoint kernels' ranges: the sizes at which a lane,
tile, tile list or ring of samples is partly filled, against the oracle,
identities, independent forward differences and the general paths."""
import numpy as np
import pytest

from paper_0909_4039_gb300 import inputs
from tests import test_gpu_adjoint as adj
from tests._common import gpu_stepper, oracle_problem, rel_l2

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12
FP32_TOL = 1e-4


def _w(Nr, Nth, m=2, r0=8.0):
    return inputs.Workload("edge", s=-2, m=m, a=0.7, Nr=Nr, Ntheta=Nth, rs_min=-60.0, rs_max=240.0, steps=0, r0=r0,
                           amp=0.8 - 0.3j, sig_r=0.9, sig_th=0.3, rs_ext=150.0)


@pytest.mark.parametrize("Nth", [129, 200, 256, 257, 300])
def test_adjoint_step_fp64_wide_rows(Nth):
    """The FP64 adjoint's row segments of 8 (128 < Ntheta <= 256, partly
    filled and full) and 32, and rows longer than the thread block
    (Ntheta > 256), where the source derivatives read columns that other
    threads then overwrite: spin term against differences of the step, taped
    against recomputed."""
    adj.test_one_step_spin_term_against_step_differences(False, 2, Nth)
    adj.test_tape_step_and_adjoint_equal_recompute(False, 2, Nth, "fp64")


@pytest.mark.parametrize("precision,Nth", [("fp64", 127), ("fp64", 129), ("fp64", 200), ("fp64", 257),
                                            ("fp32", 129), ("fp32", 132), ("fp32", 200), ("fp32", 256)])
def test_row_segments_against_oracle_and_tile_shapes(precision, Nth):
    """Row segments that are partly filled (FP64 planes; FP32 packed pairs for
    128 < Ntheta <= 256 in multiples of 4, and 129 beside them) against the
    oracle, in tiles that end within the grid; every tile height and number
    of steps per launch gives the same bits."""
    from oracle import oracle as O
    w = _w(310, Nth)
    u0, n, got = inputs.random_state(w.Nr, Nth, seed=5), 7, []
    for tr, ks in [(None, None), (1, 1), (5, 2), (6, 3), (9, 1)]:
        st = gpu_stepper(w, precision, wave_capacity=n + 1)
        if tr is not None:
            st.set_tiling(tr, ks)
        st.set_state(u0, 0)
        st.step(n)
        got.append((st.get_state(), st.waveform(0, n + 1)))
        st.close()
    uo, ho = O.run(oracle_problem(w), u0, n)
    tol = FP64_TOL if precision == "fp64" else FP32_TOL
    assert rel_l2(got[0][0], uo) <= tol and rel_l2(got[0][1], ho) <= tol
    for u, h in got[1:]:
        assert np.array_equal(u, got[0][0]) and np.array_equal(h, got[0][1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ks", [1, 2, 3])
def test_samples_of_long_calls_and_short_rings(precision, ks):
    """Waveform samples are the same from one call (graph replays, several
    sampling launches, a remainder), from calls of one to a few steps, and from
    a ring shorter than the call."""
    w = _w(90, 24)
    u0, n = inputs.random_state(w.Nr, 24, seed=9), 331
    def run(cap, calls):
        st = gpu_stepper(w, precision, wave_capacity=cap)
        st.set_tiling(16, ks)
        st.set_state(u0, 0)
        for k in calls:
            st.step(k)
        h = st.waveform(max(0, n + 1 - cap), min(cap, n + 1), rows=True)
        u = st.get_state()
        st.close()
        return u, np.asarray(h[0]), np.asarray(h[1])
    one, many, short = run(n + 1, [n]), run(n + 1, [1, 129, 2, 3, 4] * 2 + [53]), run(50, [n])
    # (noise on this coarse grid grows past FP32's range in some rows of the state)
    assert np.isfinite(one[1]).all() and np.isfinite(one[2]).all()
    assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(one, many))
    assert np.array_equal(short[0], one[0], equal_nan=True)
    assert np.array_equal(short[1], one[1][-50:]) and np.array_equal(short[2], one[2][-50:])


@pytest.mark.parametrize("precision,Nr,Nth,tr", [("fp32", 4000, 100, 12), ("fp32", 4000, 128, 12), ("fp32", 2000, 200, 12),
                                                 ("fp64", 4500, 64, 28)])
def test_batch_of_many_tiles_ends_in_half_tiles(precision, Nr, Nth, tr):
    """A batch of more than two waves of tiles takes its last rows in tiles of
    half the height: more tiles than rows / height, the same bits as alone."""
    from paper_0909_4039_gb300 import teuk
    ws = [_w(Nr, Nth, m, r0) for m, r0 in ((2, 8.0), (1, 60.0))]
    u0, n, alone = [inputs.random_state(Nr, Nth, seed=20 + k) for k in range(2)], 5, []
    for w, u in zip(ws, u0):
        st = gpu_stepper(w, precision, wave_capacity=n + 1)
        st.set_state(u, 0)
        st.step(n)
        alone.append((st.get_state(), st.waveform(0, n + 1)))
        st.close()
    sts = [gpu_stepper(w, precision, wave_capacity=n + 1) for w in ws]
    b = teuk.Batch(sts)
    b.set_tiling([tr, tr])
    assert b.tiling()["total_tiles"] > 2 * -(-Nr // tr)
    for st, u in zip(sts, u0):
        st.set_state(u, 0)
    b.step(n)
    b.synchronize()
    for st, (u, h) in zip(sts, alone):
        assert np.array_equal(st.get_state(), u) and np.array_equal(st.waveform(0, n + 1), h)
    b.close()
    for st in sts:
        st.close()


@pytest.mark.parametrize("precision,ks", [("fp64", 1), ("fp32", 3)])
def test_steps_under_stream_capture(precision, ks):
    """Steps captured into the caller's graph (dependent launches become graph
    edges) and replayed once give the state and samples of plain steps."""
    import torch
    w = _w(200, 32)
    u0, n = inputs.random_state(w.Nr, 32, seed=3), 7
    res = []
    for captured in (False, True):
        st = gpu_stepper(w, precision, wave_capacity=n + 1)
        st.set_tiling(16, ks)
        st.set_state(u0, 0)
        st.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st.stream):
                st.step(n)
            with torch.cuda.stream(st.stream):
                g.replay()
        else:
            st.step(n)
        st.synchronize()
        res.append((st.get_state(), st.waveform(0, n + 1)))
        st.close()
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("widths", [(256, 250), (255, 252), (256, 129)])
def test_fp32_batch_of_packed_and_scalar_widths(widths):
    """FP32 rows of 129 to 256 points run on packed pairs alone where Ntheta is
    a multiple of 4 and in the scalar kernel otherwise; a batch that mixes the
    two runs the scalar kernel for all of them.  At the default heights, at low
    ones and with one step a launch, each instance gets its solo run's bits."""
    from oracle import oracle as O
    from paper_0909_4039_gb300 import teuk
    ws = [_w(310 + 7 * k, Nth, 2 - k, 8.0 + k) for k, Nth in enumerate(widths)]
    u0, n, alone = [inputs.random_state(w.Nr, w.Ntheta, seed=40 + k) for k, w in enumerate(ws)], 6, []
    for w, u in zip(ws, u0):
        st = gpu_stepper(w, "fp32", wave_capacity=n + 1)
        st.set_state(u, 0)
        st.step(n)
        alone.append((st.get_state(), st.waveform(0, n + 1)))
        st.close()
        uo, ho = O.run(oracle_problem(w), u, n)
        assert rel_l2(alone[-1][0], uo) <= FP32_TOL and rel_l2(alone[-1][1], ho) <= FP32_TOL
    sts = [gpu_stepper(w, "fp32", wave_capacity=n + 1) for w in ws]
    b = teuk.Batch(sts)
    for heights, ks in ((None, None), ([4, 4], 2), ([1, 12], 2), ([6, 3], 1)):
        if heights:
            b.set_tiling(heights, ks)
        for st, u in zip(sts, u0):
            st.set_state(u, 0)
        b.step(n)
        b.synchronize()
        for st, (u, h) in zip(sts, alone):
            assert np.array_equal(st.get_state(), u) and np.array_equal(st.waveform(0, n + 1), h)
    b.close()
    for st in sts:
        st.close()


@pytest.mark.parametrize("Nth,tall", [(132, (97, 94, 92)), (200, (64, 61, 59)), (250, (51, 48, 46))])
def test_fp32_tall_tiles_of_paired_widths(Nth, tall):
    """Heights beyond a pair tile's (and, at 250 points, the tallest plain tiles):
    accepted for a lone state with one, two and three steps a launch and in a
    batch, with the bits of the default tiles."""
    from paper_0909_4039_gb300 import teuk
    w, n, got = _w(330, Nth), 7, []
    u0 = inputs.random_state(w.Nr, Nth, seed=50)
    for ks, tr in [(None, None), *enumerate(tall, 1)]:
        st = gpu_stepper(w, "fp32", wave_capacity=n + 1)
        if tr:
            st.set_tiling(tr, ks)
            assert st.tiling()["tile_rows"] == tr
        st.set_state(u0, 0)
        st.step(n)
        got.append((st.get_state(), st.waveform(0, n + 1)))
        st.close()
    st = gpu_stepper(w, "fp32", wave_capacity=n + 1)
    b = teuk.Batch([st])
    for ks in (2, 1):
        # (the batched kernel's parameters take a kilobyte of their own)
        b.set_tiling([tall[ks - 1] - 1], ks)
        st.set_state(u0, 0)
        b.step(n)
        b.synchronize()
        got.append((st.get_state(), st.waveform(0, n + 1)))
    b.close()
    st.close()
    for u, h in got[1:]:
        assert np.array_equal(u, got[0][0]) and np.array_equal(h, got[0][1])


def test_batch_whose_tiles_fill_their_last_wave_keeps_them_whole():
    """600 FP64 tiles on 152 SMs (3.95 waves): half-height tiles at the end of the
    list would end a third of a tile later, so every tile has the full height."""
    import torch
    from paper_0909_4039_gb300 import teuk
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the tile counts are for 152 SMs")
    sts = [gpu_stepper(_w(3000, 200, m, r0), "fp64", wave_capacity=4) for m, r0 in ((2, 8.0), (1, 9.0), (3, 7.0), (4, 12.0))]
    b = teuk.Batch(sts)
    b.set_tiling([20] * 4, 2)
    assert b.tiling()["total_tiles"] == 600
    b.close()
    for st in sts:
        st.close()


@pytest.mark.parametrize("precision,Nr,Nth,tiling", [("fp32", 330, 130, None), ("fp32", 330, 200, None), ("fp32", 330, 256, (7, 1)),
                                                     ("fp32", 700, 300, (2, 2)), ("fp32", 700, 300, (2, 1)),
                                                     ("fp64", 330, 300, None)])
def test_samples_of_short_calls_on_wide_rows(precision, Nr, Nth, tiling):
    """Calls of one to a few steps on rows of more than 128 points, whose tiles
    sample their own steps where a sampling launch would lengthen the call (FP32:
    one step up to 256 points; up to four steps above, on grids of more than two
    tiles per SM), give the samples, rows and state of one call; so do the calls
    of a batch of one such instance."""
    from paper_0909_4039_gb300 import teuk
    w = _w(Nr, Nth)
    u0, n, res = inputs.random_state(Nr, Nth, seed=60), 14, []
    calls = [1, 1, 2, 3, 1, 4, 2]
    for k, plan in enumerate(([n], calls, calls)):
        st = gpu_stepper(w, precision, wave_capacity=n + 1)
        if tiling and k < 2:
            st.set_tiling(*tiling)
        st.set_state(u0, 0)
        b = teuk.Batch([st]) if k == 2 else None
        for c in plan:
            (b or st).step(c)
        if b:
            b.synchronize()
            b.close()
        h, rows = st.waveform(0, n + 1, rows=True)
        res.append((st.get_state(), np.asarray(h), np.asarray(rows)))
        st.close()
    for r in res[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(r, res[0]))
