"""The warp and medium paths' sieve, the joined count-and-rows graph and the
block-tile list order, at the sizes where they can go wrong: edges of the rounds
of 32 hits and of the paths' limits, cells that wrap around the maps, odd
coordinates, stations at the end of the hit arrays, more triples than wait for
their fits, lists beyond the sort.  Everything is a whole number and is compared
with the oracle for equality."""
import numpy as np
import pytest

from gpu_helpers import assert_same, gpu_select
from helpers import layer_z, make_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_1810_11966_gb300 as jp
    jp.load(build_if_missing=True)
    return jp


def _event(rng, sizes, spread=0.02, centre=(0.2, -0.1), jitter=0.0):
    """One event with the given hits per layer, all within `spread` of one slope,
    so that cells collide and triplets abound; z may vary inside a layer."""
    ev = []
    for z0, n in zip(layer_z(len(sizes) // 3), sizes):
        z = z0 + jitter * rng.uniform(-1, 1, n)
        s = rng.uniform(-spread, spread, (n, 2)) + centre
        ev.append(list(zip(s[:, 0] * z, s[:, 1] * z, z)))
    return ev


def _check(lib, oracle_mod, b, S, t=0.25, modes=(0, 1), forms=("plain", "batched"), label=""):
    for mode in modes:
        ref = oracle_mod.run(oracle_mod.params(S, mode, t_xz=t, t_yz=t), b, n_threads=8)
        assert ref["status"] == 0
        ctx = lib.Context(lib.params(S, mode, t_xz=t, t_yz=t))
        for form in forms:
            assert_same(gpu_select(ctx, b, form=form), ref, b["n_events"] * S, label=f"{label} mode{mode} {form} t={t}")
        ctx.close()


# hits of the three layers of a station: edges of a round, of 64, 128 and 192 hits
# per layer, and of 384 per station; then those of the medium path (384, 960)
WARP = [(1, 1, 1), (31, 32, 33), (0, 5, 5), (5, 0, 5), (5, 5, 0), (63, 64, 65), (64, 64, 64), (65, 1, 128),
        (128, 128, 128), (129, 127, 128), (1, 192, 191), (192, 96, 96), (96, 192, 96), (96, 96, 192), (3, 129, 2)]
MEDIUM = [(193, 1, 1), (1, 193, 1), (129, 128, 128), (255, 256, 257), (384, 384, 192), (192, 384, 384), (320, 320, 320),
          (1, 1, 384), (321, 320, 320), (385, 5, 5)]


@pytest.mark.parametrize("sizes", [WARP, MEDIUM], ids=["warp", "medium"])
def test_layer_sizes(lib, oracle_mod, sizes):
    rng = np.random.default_rng(11)
    events = []
    for a in sizes:
        # a wide spread keeps the trigger triplets few enough for the path's list
        wide = 0.2 if max(a) > 40 else 0.05
        events.append(_event(rng, list(a) + list(sizes[rng.integers(len(sizes))]), spread=wide, centre=(0.0, 0.0)))
        events.append(_event(rng, list(a) + [4, 3, 4], spread=wide, centre=(0.0, 0.0), jitter=3.0))
    _check(lib, oracle_mod, make_batch(events, 2), 2)


@pytest.mark.parametrize("t", [0.0, 1e-9, 1e-4, 4.0, 400.0, 1e30])
def test_windows_from_points_to_everything(lib, oracle_mod, t):
    # cells from far below to far beyond the spread of the hits: they wrap around
    # the maps many times, or all hits share one
    rng = np.random.default_rng(12)
    events = [_event(rng, [12, 9, 11, 10, 12, 9], spread=0.3, centre=(0.0, 0.0)) for _ in range(20)]
    events += [_event(rng, [2, 200, 2, 3, 3, 3], spread=0.3, centre=(0.0, 0.0))]
    for slope in (0.1, -0.35, 3.0, 4e4):  # straight tracks: pass whatever the cut
        events.append([[(slope * z, -0.5 * slope * z, z)] * 2 for z in layer_z(2)])
    _check(lib, oracle_mod, make_batch(events, 2), 2, t=t)


def test_odd_coordinates_among_ordinary_hits(lib, oracle_mod):
    rng = np.random.default_rng(13)
    odd = [np.nan, np.inf, -np.inf, 1e-42, 3e38, 0.0]
    events = []
    for n in (3, 33, 64, 100, 150, 250):
        for v in odd:
            ev = _event(rng, [n] * 6, spread=0.25, centre=(0.0, 0.0))
            layer, at, coord = rng.integers(6), rng.integers(n), rng.integers(3)
            h = list(ev[layer][at])
            h[coord] = v if coord < 2 or v > 0 or np.isnan(v) else 1e-42
            ev[layer][at] = tuple(h)
            events.append(ev)
    _check(lib, oracle_mod, make_batch(events, 2), 2)


@pytest.mark.parametrize("n_events", [1, 2, 33])
def test_last_stations_of_the_arrays(lib, oracle_mod, n_events):
    # every station lies so close to the end of the arrays that full rounds would leave them
    rng = np.random.default_rng(14)
    events = [_event(rng, [3, 1, 2, 2, 3, 1], spread=0.01) for _ in range(n_events)]
    _check(lib, oracle_mod, make_batch(events, 2), 2)


@pytest.mark.parametrize("m", [4, 5, 12, 30])
def test_more_triples_than_wait_for_a_fit(lib, oracle_mod, m):
    # m equal hits per layer of a non-trigger station: m^3 triplets of one unit (up
    # to 27 000) beside few, no or (trigger station) too many trigger triplets
    zl = layer_z(3)
    line = lambda z, n: [(0.1 * z, 0.2 * z, z)] * n  # noqa: E731
    events = []
    for last in (0, 1, 2, 4):
        for big in (m, 0):
            events.append([line(z, big if l < 3 else 2 if l < 6 else last) for l, z in enumerate(zl)])
    pad = _event(np.random.default_rng(15), [200, 3, 3] * 3, spread=0.3, centre=(-0.2, 0.1))
    events += [[a + b for a, b in zip(ev, pad)] for ev in events]  # the same on the medium path
    _check(lib, oracle_mod, make_batch(events, 3), 3)


def test_rows_behind_the_count(lib, oracle_mod, synth_mod):
    # untimed batched runs scatter the rows behind the count: too small a buffer,
    # the same buffer again, and a record that overflows
    b = synth_mod.generate("lognormal_timeslices", 0, 1200)
    ref = oracle_mod.run(oracle_mod.params(4, 1, t_xz=0.25), b, n_threads=8)
    need = ref["trip_needed"]
    for record_cap in (-1, max(need // 3, 1)):
        ctx = lib.Context(lib.params(4, 1, t_xz=0.25))
        tu = lib.jpsi_get_tuning(ctx.ctx)
        tu.record_cap = record_cap
        assert lib.jpsi_set_tuning(ctx.ctx, tu) == lib.JPSI_OK
        for _ in range(2):
            g = gpu_select(ctx, b, capacity=need - 1)
            assert g["status"] == lib.JPSI_ECAPACITY and g["trip_needed"] == need
            assert np.array_equal(g["trip_off"], ref["trip_off"])
            assert np.array_equal(g["track_counts"], ref["track_counts"])
            assert_same(gpu_select(ctx, b, capacity=need), ref, 4800)
            assert_same(gpu_select(ctx, b, capacity=3 * need), ref, 4800)
        ctx.close()


@pytest.mark.parametrize("n_events", [2, 8192, 8193])
def test_block_tile_list(lib, oracle_mod, n_events):
    # every event on the block tile: the longest list that is ordered, and one more
    rng = np.random.default_rng(16)
    events = [_event(rng, list(rng.integers(2, 6, 6)), spread=0.02) for _ in range(n_events)]
    b = make_batch(events, 2)
    ref = oracle_mod.run(oracle_mod.params(2, 1, t_xz=0.25), b, n_threads=8)
    ctx = lib.Context(lib.params(2, 1, t_xz=0.25))
    tu = lib.jpsi_get_tuning(ctx.ctx)
    tu.small_layer_cap = tu.medium_layer_cap = 1
    assert lib.jpsi_set_tuning(ctx.ctx, tu) == lib.JPSI_OK
    assert_same(gpu_select(ctx, b), ref, 2 * n_events)


@pytest.mark.parametrize("n_events", [4255, 4256, 8511, 8512, 8513, 17025])
def test_grab_sizes(lib, oracle_mod, n_events):
    # around one and two grabs per resident warp
    rng = np.random.default_rng(17)
    base = [_event(rng, list(rng.integers(0, 5, 3)), spread=0.01) for _ in range(64)]
    b = make_batch([base[k % 64] for k in range(n_events)], 1)
    _check(lib, oracle_mod, b, 1, modes=(1,), forms=("batched",))


def test_many_stations(lib, oracle_mod):
    # 10 and 16 stations: offsets beyond one per lane
    rng = np.random.default_rng(18)
    for S in (9, 10, 16):
        sz = tuple(130.0 + 35.0 * s for s in range(S))
        events = []
        for _ in range(12):
            ev = []
            for z0 in layer_z(S, station_z=sz):
                ev.append([(0.1 * z0 + rng.normal(0, 0.1), 0.2 * z0 + rng.normal(0, 0.1), z0) for _ in range(3)]
                          + [(rng.uniform(-60, 60), rng.uniform(-60, 60), z0) for _ in range(rng.integers(0, 9))])
            events.append(ev)
        _check(lib, oracle_mod, make_batch(events, S), S)
