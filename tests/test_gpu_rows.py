"""The site-per-lane sweep kernel (the choice of MUCA_RES_AUTO) against the
oracle, bit for bit: every way a row is laid out on a warp (one segment, rows
that are no multiple of 4, the last length of each shared-memory row width, two
to four segments with full and ragged last ones), the hot regime in
which a row takes many passes, narrow windows, and checkpoints between its
lattice layout and the walker-minor one."""
import numpy as np
import pytest

import oracle
from paper_1502_07214_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def muca():
    from paper_1502_07214_gb300 import muca as m

    return m


def run_against_oracle(L, T, W, lnW, n, bonds=None, e_min=0, e_max=None, spins0=None,
                       walkers=None):
    V = L ** 3
    e_max = V if e_max is None else e_max
    c = muca().Context([{"L": L, "T": T, "n_walkers": W, "e_min": e_min, "e_max": e_max}], seed=L)
    if spins0 is not None:
        c.set_state(0, spins0)
    if bonds is not None:
        c.set_bonds(0, bonds)
    assert c.get_config(0)[0] == (muca().RES_ROWS if bonds is None else muca().RES_BONDS)
    c.set_lnW(0, lnW)
    c.reserve_timeseries(n)
    c.sweep_iter(n, record=True)
    spins, tal = c.get_state(0)
    ts, H = c.get_timeseries(0), c.get_hist(0)
    c.check_tallies()
    c.close()
    jmax = None if bonds is None else int(np.abs(bonds).max())
    thr = (oracle.build_table(L, T, e_min, e_max, lnW) if bonds is None else
           oracle.build_table_bonds(L, T, jmax, e_min, e_max, lnW))
    for w in walkers or range(W):
        sp = oracle.init_spins(L, L, w) if spins0 is None else spins0[w].copy()
        if bonds is None:
            t = oracle.energies(L, sp).astype(np.int32)
            ref = oracle.sweeps(L, e_min, e_max, thr, L, w, 0, n, sp, t, record=True)
        else:
            t = oracle.energies_bonds(L, sp, bonds).astype(np.int32)
            ref = oracle.sweeps_bonds(L, bonds, jmax, e_min, e_max, thr, L, w, 0, n, sp, t,
                                      record=True)
        assert np.array_equal(spins[w], sp) and np.array_equal(tal[w], t), w
        assert np.array_equal(ts[:, :, w], ref), w
    assert np.array_equal(H, np.bincount(ts[:, 1, :].ravel() - e_min,
                                         minlength=len(H)).astype(np.uint64))


# (L, walkers): one walker more than whole warps where several share one
@pytest.mark.parametrize("L,W", [(3, 21), (4, 17), (5, 13), (8, 9), (11, 5), (12, 7), (13, 5),
                                 (16, 5), (17, 3), (22, 3), (31, 2), (32, 3), (33, 5), (48, 5),
                                 (49, 3), (61, 3), (64, 3)])
def test_every_row_layout_under_rough_transition_weights(L, W):
    """Weights with the transition's slope and a roughness of 0.5 per bin from
    the random start: some ten accepted moves per row, whose order matters."""
    T = 1.0
    lnW = -2.944 / T * np.arange(L ** 3 + 1) + wl.random_lnW(L ** 3 + 1, L, scale=0.5)
    run_against_oracle(L, T, W, lnW, 3 if L <= 33 else 2)


@pytest.mark.parametrize("L,jj", [(33, None), (48, None), (49, None), (64, None), (40, (1, 3)),
                                  (52, (-1, 2))])
def test_long_rows_of_many_walkers(L, jj):
    """More than 608 walkers: rows beyond 32 sites in three or four segments, two
    walkers per warp (fewer walkers take two segments); sampled walkers."""
    V = L ** 3
    lnW = -1.5 * np.arange(V + 1) + wl.random_lnW(V + 1, L, scale=0.5)
    run_against_oracle(L, 3.0, 611, lnW, 2, walkers=[0, 1, 2, 305, 609, 610],
                       bonds=None if jj is None else wl.random_bonds(L, jj[0], jj[1], seed=L))


@pytest.mark.parametrize("L,W,jj", [(3, 12, (1, 3)), (7, 6, (-1, 1)), (12, 5, (2, 8)),
                                    (18, 3, (5, 3)), (32, 2, (0, 2)), (36, 3, (-3, 1))])
def test_couplings_in_every_row_layout(L, W, jj):
    lnW = -1.5 * np.arange(L ** 3 + 1) + wl.random_lnW(L ** 3 + 1, L, scale=0.5)
    run_against_oracle(L, 3.0, W, lnW, 2, bonds=wl.random_bonds(L, jj[0], jj[1], seed=L))


@pytest.mark.parametrize("e_min,e_max", [(256, 256), (250, 262), (0, 300), (200, 512)])
def test_narrow_windows(e_min, e_max):
    L, W = 8, 6
    rng = np.random.default_rng(4)
    spins = np.zeros((W, L ** 3), dtype=np.int8)
    for w in range(W):
        at = rng.permutation(L ** 3)[:256]
        spins[w, at] = rng.choice(np.array([-1, 1], dtype=np.int8), 256)
    run_against_oracle(L, 1.4182, W, wl.random_lnW(e_max - e_min + 1, 3), 20, e_min=e_min,
                       e_max=e_max, spins0=spins)


@pytest.mark.parametrize("L", [6, 20, 34])
def test_checkpoints_cross_lattice_layouts(L, tmp_path):
    """A file written from one layout continues bit-identically in the other."""
    g = [{"L": L, "T": 1.4182, "n_walkers": 5}]
    a = muca().Context(g, seed=7)
    b = muca().Context(g, seed=7, residency=muca().RES_GLOBAL, walkers_per_block=32)
    assert a.get_config(0)[0] == muca().RES_ROWS and b.get_config(0)[0] == muca().RES_GLOBAL
    a.sweep_iter(3)
    pa, pb = str(tmp_path / "a"), str(tmp_path / "b")
    a.checkpoint(pa)
    b.restore(pa)
    b.sweep_iter(2)
    b.checkpoint(pb)
    a.sweep_iter(2)
    want = a.get_state(0)
    a.restore(pb)
    for c in (a, b):
        got = c.get_state(0)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        c.close()


def _groups_against_the_general_path(groups, bonds, n):
    """All groups of one context on the site-per-lane kernel, and on the
    lanes-per-walker kernel: state, histogram and series bit for bit."""
    out = []
    for kw in ({}, {"residency": muca().RES_GLOBAL, "walkers_per_block": 32}):
        c = muca().Context(groups, seed=9, **kw)
        for g, s in enumerate(groups):
            V = s["L"] ** 3
            if g in bonds:
                c.set_bonds(g, bonds[g])
            elif not kw:
                assert c.get_config(g)[0] == muca().RES_ROWS
            c.set_lnW(g, -1.5 * np.arange(V + 1) + wl.random_lnW(V + 1, g, scale=0.3))
        c.reserve_timeseries(n)
        c.sweep_iter(n, record=True)
        out.append([(c.get_state(g), c.get_hist(g), c.get_timeseries(g))
                    for g in range(len(groups))])
        c.check_tallies()
        c.close()
    for g, (a, b) in enumerate(zip(*out)):
        assert np.array_equal(a[0][0], b[0][0]) and np.array_equal(a[0][1], b[0][1]), g
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2]), g


@pytest.mark.parametrize("n_groups", [2, 5, 127, 128, 129, 300])
def test_many_groups_share_launches(n_groups):
    """One launch takes 128 groups: row lengths, walkers per warp and block
    counts that differ from group to group."""
    rng = np.random.default_rng(n_groups)
    groups = [{"L": int(L), "T": float(T), "n_walkers": int(W)} for L, T, W in
              zip(rng.integers(3, 10, n_groups), rng.choice([0.9, 1.4182, 3.0], n_groups),
                  rng.integers(1, 40, n_groups))]
    _groups_against_the_general_path(groups, {}, 3)


def test_groups_of_every_kind_in_one_context():
    """Row widths, segment counts, couplings and L = 2 (no site-per-lane rows)."""
    Ls = [3, 16, 17, 32, 33, 48, 49, 64, 16, 20, 33, 3, 12, 48, 50]
    groups = [{"L": L, "T": 1.4182, "n_walkers": 3 + i} for i, L in enumerate(Ls)]
    groups.append({"L": 36, "T": 1.4182, "n_walkers": 620})
    bonds = {i: wl.random_bonds(groups[i]["L"], 5, 3, seed=i) for i in (1, 8, 9, 10, 14)}
    _groups_against_the_general_path(groups, bonds, 2)


def test_many_small_groups_run_side_by_side():
    """256 groups of 32 walkers fill a sixth of the chip: a sweep of them takes
    little longer than one of 24 such groups (measured 1.5 times; 7.8 times when
    groups beyond the 32nd waited for one another)."""
    import time

    t = []
    for k in (24, 256):
        c = muca().Context([{"L": 8, "T": 1.4182, "n_walkers": 32}] * k, seed=3)
        c.sweep_iter(50)
        c.sync()
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            c.sweep_iter(200)
            c.sync()
            best = min(best, time.perf_counter() - t0)
        t.append(best)
        c.close()
    assert t[1] <= 4 * t[0], t


@pytest.mark.parametrize("L,jj", [(33, None), (41, None), (48, None), (40, (1, 3)), (45, (-1, 2))])
def test_three_segments_beyond_one_wave_of_warps(L, jj):
    """Rows of 33 to 48 sites of more walkers than the GPU holds warps (16 per SM)
    are cut into three segments, two walkers per warp; sampled walkers."""
    V, W = L ** 3, 16 * torch.cuda.get_device_properties(0).multi_processor_count + 3
    c = muca().Context([{"L": L, "T": 3.0, "n_walkers": n} for n in (W - 3, W)], seed=1)
    assert [c.get_config(g)[2] for g in (0, 1)] == [(L + 2) // 3] * 2  # together
    c.close()
    c = muca().Context([{"L": L, "T": 3.0, "n_walkers": W - 3}], seed=1)
    assert c.get_config(0)[1:] == (1, (L + 1) // 2)
    c.close()
    lnW = -1.5 * np.arange(V + 1) + wl.random_lnW(V + 1, L, scale=0.5)
    run_against_oracle(L, 3.0, W, lnW, 2, walkers=[0, 1, 2, W // 2, W - 2, W - 1],
                       bonds=None if jj is None else wl.random_bonds(L, jj[0], jj[1], seed=L))


@pytest.mark.parametrize("L,W", [(5, 7), (12, 3), (13, 5), (16, 3), (20, 3), (32, 2), (34, 3),
                                 (47, 2), (52, 2), (62, 2), (40, 2501)])
def test_couplings_with_an_explicit_residency(L, W):
    """A group whose lattice was laid out for another kernel (walker-minor words)
    and then gets couplings: planes pass through shared memory word by word."""
    V, n = L ** 3, 3
    J = wl.random_bonds(L, -2, 3, seed=L)
    lnW = -1.5 * np.arange(V + 1) + wl.random_lnW(V + 1, L, scale=0.5)
    c = muca().Context([{"L": L, "T": 3.0, "n_walkers": W}], seed=L, residency=muca().RES_GLOBAL,
                       walkers_per_block=32)
    c.set_bonds(0, J)
    c.set_lnW(0, lnW)
    c.reserve_timeseries(n)
    c.sweep_iter(n, record=True)
    spins, tal = c.get_state(0)
    ts = c.get_timeseries(0)
    c.check_tallies()
    c.close()
    thr = oracle.build_table_bonds(L, 3.0, 3, 0, V, lnW)
    for w in sorted({0, 1, W // 2, W - 1}):
        sp = oracle.init_spins(L, L, w)
        t = oracle.energies_bonds(L, sp, J).astype(np.int32)
        ref = oracle.sweeps_bonds(L, J, 3, 0, V, thr, L, w, 0, n, sp, t, record=True)
        assert np.array_equal(spins[w], sp) and np.array_equal(tal[w], t), w
        assert np.array_equal(ts[:, :, w], ref), w


@pytest.mark.parametrize("L,W", [(2, 40), (3, 33), (8, 20), (22, 5), (48, 3), (64, 2)])
def test_a_reported_configuration_can_be_given_again(L, W):
    """A program that keeps get_config's result and pins it later."""
    groups = [{"L": L, "T": 1.4182, "n_walkers": W}]
    a = muca().Context(groups, seed=4)
    cfg = a.get_config(0)
    b = muca().Context(groups, seed=4, residency=cfg[0], walkers_per_block=cfg[1],
                       lanes_per_walker=cfg[2])
    assert b.get_config(0) == cfg
    for c in (a, b):
        c.run_graph(1, 4)
    assert np.array_equal(a.get_state(0)[0], b.get_state(0)[0])
    assert np.array_equal(a.get_lnW(0), b.get_lnW(0))
    a.close()
    b.close()
    for bad in (muca().RES_BONDS, 7, -1):
        with pytest.raises(muca().MucaError) as e:
            muca().Context(groups, residency=bad)
        assert e.value.code == muca().ERR_INVALID_ARG
    with pytest.raises(muca().MucaError):
        muca().Context(groups, residency=muca().RES_ROWS, lanes_per_walker=33)


def test_lattices_that_fit_only_with_packed_rows():
    """Groups whose lattices fit the free memory with packed rows, not with rows
    padded for 16-byte copies, are accepted, and swept in that layout."""
    Ls = [17, 13, 22, 34, 50] + [17] * 8
    groups = [{"L": L, "T": 3.0, "n_walkers": 10000 if i > 4 else 3} for i, L in enumerate(Ls)]
    packed = sum(s["n_walkers"] * s["L"] ** 2 * ((s["L"] + 3) // 4) * 4 for s in groups)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - packed - (100 << 20), dtype=torch.uint8,
                          device="cuda")
    try:
        c = muca().Context(groups, seed=6)
        out = []
        for g, s in enumerate(groups):
            assert c.get_config(g)[0] == muca().RES_ROWS
            V = s["L"] ** 3
            c.set_lnW(g, -1.5 * np.arange(V + 1) + wl.random_lnW(V + 1, g, scale=0.5))
        c.sweep_iter(2)
        for g in range(6):
            out.append((c.get_state(g), c.get_lnW(g), c.specs[g]["first_walker"]))
        c.check_tallies()
        c.close()
    finally:
        del ballast
        torch.cuda.empty_cache()
    for s, ((spins, tal), lnW, w0) in zip(groups, out):
        L, V = s["L"], s["L"] ** 3
        thr = oracle.build_table(L, 3.0, 0, V, lnW)
        for w in (0, 1, len(spins) - 1):
            sp = oracle.init_spins(L, 6, w0 + w)
            t = oracle.energies(L, sp).astype(np.int32)
            oracle.sweeps(L, 0, V, thr, 6, w0 + w, 0, 2, sp, t)
            assert np.array_equal(spins[w], sp) and np.array_equal(tal[w], t), (L, w)


def test_state_calls_keep_pace_with_the_walker_minor_layout(tmp_path):
    """Checkpoint, restore and tally checks of a lattice kept walker by walker (the
    file's order is walker-minor; two pieces of 64 MiB) against the same walkers
    on the walker-minor layout: the same files, and no more than twice as
    long (measured 0.03 to 1.0 times; 2.8 to 6 times when reordered on the host and
    summed by a thread per walker)."""
    import time

    g = [{"L": 48, "T": 1.4182, "n_walkers": 1024}]
    a = muca().Context(g, seed=7)
    b = muca().Context(g, seed=7, residency=muca().RES_GLOBAL, walkers_per_block=32)
    best = {}
    paths = {}
    for name, c in (("a", a), ("b", b)):
        c.sweep_iter(2)
        paths[name] = str(tmp_path / name)
        for what, f in (("checkpoint", lambda: c.checkpoint(paths[name])),
                        ("restore", lambda: c.restore(paths[name])),
                        ("check_tallies", c.check_tallies)):
            t = []
            for _ in range(4):
                t0 = time.perf_counter()
                f()
                t.append(time.perf_counter() - t0)
            best[what, name] = min(t)
    files = [open(p, "rb").read() for p in (paths["a"], paths["b"])]
    assert files[0] == files[1]
    a.restore(paths["b"])
    for x, y in zip(a.get_state(0), b.get_state(0)):
        assert np.array_equal(x, y)
    a.close()
    b.close()
    for what in ("checkpoint", "restore", "check_tallies"):
        assert best[what, "a"] <= 2 * best[what, "b"], best
