"""Beads in their bins' slots (a2): bins that hold more beads than they have
slots, runs of several steps, the sorted read-outs and saved images."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import assert_field, t2n
from paper_2607_02954_gb300 import World, step_batched, synth

pytestmark = pytest.mark.gpu


def crowded(seed, n_fil=30, B=4, H=72, W=64, at=(60.0, 68.0)):
    """n_fil short filaments within one or two 8x8 bins at the periodic corner
    and a few spread over the rest."""
    rng = np.random.default_rng(seed)
    lengths = [B] * n_fil + [9] * 5
    x, y, th = [], [], []
    for f, b in enumerate(lengths):
        h = rng.uniform(0, 2 * np.pi)
        x0, y0 = (at[0] + rng.uniform(0, 3), at[1] + rng.uniform(0, 3)) if f < n_fil else rng.uniform(10, 40, 2)
        k = np.arange(b)
        x.append(np.mod(x0 + k * np.cos(h), W))
        y.append(np.mod(y0 + k * np.sin(h), H))
        th.append(np.full(b - 1, h))
    x, y = (np.concatenate(v).astype(np.float32) for v in (x, y))
    x[x >= W] = 0
    y[y >= H] = 0
    J = sum(b - 2 for b in lengths)
    # the forces shared by the beads of a cell stay below the velocity watchdog
    p = synth.Params(k_rep=0.02 / max(1.0, n_fil / 30) ** 2, kappa=0.05 / max(1.0, n_fil / 30) ** 2)
    return synth._world("crowded", H, W, lengths, x, y, np.concatenate(th).astype(np.float32),
                        rng.uniform(-0.2, 0.2, J), np.full(J, 0.1), np.full(J, 0.02), rng.uniform(0, 1, J), params=p)


@pytest.mark.parametrize("n_fil,kw", [(7, {}), (8, {}), (9, {}), (30, {}), (200, {}),
                                      (30, dict(layers=2)), (30, dict(ib=1, mdf_iters=2))])
def test_one_step_of_crowded_bins(n_fil, kw):
    spec = crowded(n_fil, n_fil)
    for k, v in kw.items():
        setattr(spec.params, k, v)
    _, bin_w, off_w = O.cell_and_bin(spec.x, spec.y, spec.H, spec.W, 8)
    assert n_fil < 9 or np.diff(off_w).max() > 8
    ow = O.World(spec)
    st, rec = O.step(ow, ow.initial_state(), record=True)
    w = World(spec)
    w.step(1)
    assert np.array_equal(w.field("bin"), bin_w)
    off, beads = w.field("bin_off"), w.field("bin_beads")
    assert np.array_equal(off, off_w)
    for b in np.nonzero(np.diff(off_w))[0]:
        assert np.array_equal(np.sort(beads[off[b]:off[b + 1]]), np.nonzero(bin_w == b)[0])
    # the repository's per-step bound: 1e-5 of each field's scale
    assert_field("rho_s", w.field("rho_s"), t2n(rec["rho_s"]), 1e-5)
    assert_field("rho_bar", w.field("rho_bar"), t2n(rec["rho_bar"]), 1e-5)
    assert_field("fs", w.field("fs"), t2n(rec["F_s"]), 1e-5)
    assert_field("u", w.field("u"), np.moveaxis(t2n(rec["u"]), 0, -1), 1e-5)
    assert_field("disp", w.state()["disp"], t2n(st.D), 1e-5)


@pytest.mark.parametrize("steps", [1, 2, 7, 16, 35])
def test_crowded_world_alone_batched_and_stepwise(steps):
    """Runs of fused steps, single steps and a batch agree bitwise, and so do
    the read-outs after them."""
    specs = [crowded(3), synth.world_random(4, (40, 72), 5), crowded(5, n_fil=60)]
    alone, single, batch = ([World(s) for s in specs] for _ in range(3))
    for w in alone:
        w.step(steps)
    for w in single:
        for _ in range(steps):
            w.step(1)
    step_batched(batch, steps)
    for a, s, b in zip(alone, single, batch):
        want = a.state(fluid=True)
        for other in (s, b):
            got = other.state(fluid=True)
            for k in want:
                assert np.array_equal(want[k], got[k]), k
            for f in ("fel", "fs", "bin", "bin_off", "rho_s", "rho_bar", "force"):
                assert np.array_equal(a.field(f), other.field(f)), f


@pytest.mark.parametrize("steps", [0, 1, 18])
@pytest.mark.parametrize("kw", [{}, dict(layers=2), dict(ib=1, mdf_iters=1)])
def test_saved_image_restores_the_binned_beads(steps, kw):
    spec = crowded(11)
    for k, v in kw.items():
        setattr(spec.params, k, v)
    a = World(spec)
    a.step(steps)
    b = World.load(a.save(), spec)
    if steps:
        for f in ("bin", "bin_off", "rho_s", "rho_bar", "fs", "force"):
            assert np.array_equal(a.field(f), b.field(f)), f
    for w in (a, b):
        w.step(5)
    want, got = a.state(fluid=True), b.state(fluid=True)
    for k in want:
        assert np.array_equal(want[k], got[k]), k


@pytest.mark.parametrize("n", [3, 4])
def test_rewind_to_either_parity_starts_from_empty_bins(n):
    """A rollout of an odd or even number of steps, rewound and run again,
    repeats bitwise."""
    w = World(crowded(13))
    w.rollout_forward(n, 2)
    want = w.state(fluid=True)
    w.rollout_rewind()
    w.rollout_forward(n, 2)
    got = w.state(fluid=True)
    for k in want:
        assert np.array_equal(want[k], got[k]), k
    torch.cuda.synchronize()


@pytest.mark.parametrize("H,W,n_fil,B", [(96, 64, 80, 64), (256, 256, 1024, 64), (416, 704, 2288, 64), (640, 648, 2580, 64),
                                         (480, 1288, 300, 24)])
def test_wide_tile_blocks_equal_the_narrow_ones(H, W, n_fil, B):
    """Worlds on both sides of the lines where a tile's block gets wider (few
    tiles, many beads a tile) against the persistent step, whose tiles always
    take 256 threads: bitwise the same, and one step against the oracle."""
    from paper_2607_02954_gb300 import set_launch_config
    rng = np.random.default_rng(H + W)
    f = np.arange(n_fil)
    per_row = W // B
    x, y = [], []
    rows = -(-n_fil // per_row)
    x0, y0 = (f % per_row) * B + rng.uniform(0, 0.5, n_fil), (f // per_row) * H / rows + rng.uniform(0, 0.5, n_fil)
    x = np.mod(x0[:, None] + np.arange(B)[None], W).astype(np.float32).ravel()
    y = np.mod(np.repeat(y0, B), H).astype(np.float32)
    x[x >= W] = 0
    y[y >= H] = 0
    J = n_fil * (B - 2)
    spec = synth._world("wide", H, W, [B] * n_fil, x, y, np.zeros(n_fil * (B - 1), np.float32),
                        rng.normal(0, 0.1, J), np.full(J, 0.2), np.full(J, 0.01), rng.uniform(0, 1, J),
                        params=synth.Params(k_rep=0.1))
    a, b = World(spec), World(spec)
    set_launch_config([b], persistent=4)
    for w in (a, b):
        w.step(3)
    want, got = a.state(fluid=True), b.state(fluid=True)
    for k in want:
        assert np.array_equal(want[k], got[k]), k
    for k in ("fel", "fs", "rho_s", "rho_bar", "force"):
        assert np.array_equal(a.field(k), b.field(k)), k
    ow = O.World(spec)
    _, rec = O.step(ow, ow.initial_state(), record=True)
    c = World(spec)
    c.step(1)
    assert_field("rho_s", c.field("rho_s"), t2n(rec["rho_s"]), 1e-5)
    assert_field("u", c.field("u"), np.moveaxis(t2n(rec["u"]), 0, -1), 1e-5)


@pytest.mark.parametrize("lengths", [[65], [64, 65, 2], [128, 129, 7], [300, 64, 255, 256, 257, 30], [3072, 65]])
@pytest.mark.parametrize("kw", [{}, dict(pbd_order=1), dict(layers=2), dict(ib=1, mdf_iters=1)])
def test_long_filaments_beside_short_ones(lengths, kw):
    """Filaments of more than 64 beads (a block each) beside short ones (a
    warp each): one step against the oracle, and a batch against each alone."""
    H, W = (128, 3200) if max(lengths) > 512 else (96, 320)
    rng = np.random.default_rng(sum(lengths))
    x = np.concatenate([2.0 + np.arange(b) + rng.uniform(0, 0.4) for b in lengths]).astype(np.float32)
    y = np.concatenate([np.full(b, 5.0 + 12.0 * f) for f, b in enumerate(lengths)]).astype(np.float32)
    E, J = sum(b - 1 for b in lengths), sum(b - 2 for b in lengths)
    spec = synth._world("long", H, W, lengths, x, y, np.zeros(E, np.float32), rng.normal(0, 0.1, J), np.full(J, 0.2),
                        np.full(J, 0.01), rng.uniform(0, 1, J), params=synth.Params(**kw))
    spec = synth.with_observables(spec, 3)
    ow = O.World(spec)
    st, rec = O.step(ow, ow.initial_state(), record=True)
    a = World(spec)
    a.step(1)
    assert_field("theta", a.state()["theta"], t2n(st.theta), 1e-6)
    assert_field("disp", a.state()["disp"], t2n(st.D), 1e-5)
    assert_field("fel", a.field("fel"), t2n(rec["F_el"]), 1e-5)
    # beside a world whose longest filament asks for another width of block
    other = synth.with_observables(synth.world_random(4, (40, 240), 2, lengths=[5, 200]), 4)
    batch = [World(other), World(spec), World(other)]
    step_batched(batch, 4)
    b = World(spec)
    b.step(4)
    want, got = b.state(fluid=True), batch[1].state(fluid=True)
    for k in want:
        assert np.array_equal(want[k], got[k]), k
    assert b.observables() == batch[1].observables()


@pytest.mark.parametrize("m", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("steps", [1, 2, 5, 18])
def test_direct_forcing_runs_alone_batched_and_mixed(m, steps):
    """The fused sequence of a direct-forcing world (odd and even numbers of
    passes), the unfused one it takes beside a penalty world, and single steps:
    bitwise the same, read-outs included."""
    p = dict(ib=1, mdf_iters=m)
    spec = synth.world_random(21, (72, 136), 9)
    spec.params = synth.Params(**p)
    spec = synth.with_observables(spec, 5)
    dense = crowded(17, n_fil=60)
    dense.params.ib, dense.params.mdf_iters = 1, m
    penalty = synth.world_random(22, 64, 4)
    for sp in (spec, dense):
        a, s, b, c = (World(sp) for _ in range(4))
        a.step(steps)
        for _ in range(steps):
            s.step(1)
        step_batched([b, World(sp)], steps)        # a batch of the same coupling
        step_batched([c, World(penalty)], steps)   # a mixed one
        want = a.state(fluid=True)
        for other in (s, b, c):
            got = other.state(fluid=True)
            for k in want:
                assert np.array_equal(want[k], got[k]), k
            for f in ("fel", "fs", "ubead", "u", "force", "bin", "bin_off", "rho_s", "rho_bar"):
                assert np.array_equal(a.field(f), other.field(f)), f
            assert a.observables() == other.observables()


@pytest.mark.parametrize("H,W,n_fil", [(64, 96, 20), (256, 512, 500), (520, 1288, 2000)])
def test_direct_forcing_tile_widths(H, W, n_fil):
    """One step of direct forcing with tile blocks of 1024, 512 and 256
    threads, some tiles holding more beads than one list, against the oracle."""
    rng = np.random.default_rng(H)
    B = 40
    x = np.concatenate([rng.uniform(0, W) + np.arange(B) for _ in range(n_fil)]) % W
    y = np.repeat(rng.uniform(0, H / 2, n_fil), B)
    x, y = x.astype(np.float32), y.astype(np.float32)
    x[x >= W] = 0
    J = n_fil * (B - 2)
    spec = synth._world("mdf", H, W, [B] * n_fil, x, y, np.zeros(n_fil * (B - 1), np.float32), rng.normal(0, 0.1, J),
                        np.zeros(J), np.zeros(J), np.zeros(J), params=synth.Params(ib=1, mdf_iters=2, k_rep=0.01))
    ow = O.World(spec)
    st, rec = O.step(ow, ow.initial_state(), record=True)
    w = World(spec)
    w.step(1)
    assert_field("u", w.field("u"), np.moveaxis(t2n(rec["u"]), 0, -1), 1e-5)
    assert_field("force", w.field("force"), np.moveaxis(t2n(rec["F"]), 0, -1), 1e-5)
    assert_field("ubead", w.field("ubead"), t2n(rec["U"]), 1e-5)


@pytest.mark.parametrize("kw", [{}, dict(layers=2), dict(ib=1, mdf_iters=1)])
def test_a_crowd_that_outgrows_its_bins_slots(kw):
    """A crowd carried across bins by the flow: between two layouts of the
    slots its beads find the new bins' slots full.  One run, single steps and
    a batch agree bitwise, and 12 steps agree with the oracle."""
    spec = crowded(31, n_fil=40, at=(20.0, 20.0))
    for k, v in kw.items():
        setattr(spec.params, k, v)
    cx = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
    cy = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]
    wt = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    ux, uy = 0.3, 0.1
    cu = cx * ux + cy * uy
    spec.f0 = np.broadcast_to(wt * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy)),
                              (9, spec.H, spec.W)).astype(np.float32)
    _, _, off0 = O.cell_and_bin(spec.x, spec.y, spec.H, spec.W, 8)
    room = (np.diff(off0) * 5 // 4 + 16 + 7) // 8 * 8
    a, s, b = (World(spec) for _ in range(3))
    for _ in range(12):
        s.step(1)
    assert (np.diff(s.field("bin_off")) > room).any()   # some bin outgrew the slots its first count gave it
    a.step(12)
    other = World(synth.world_random(4, (40, 72), 5))
    step_batched([b, other], 12)
    want = a.state(fluid=True)
    for w in (s, b):
        got = w.state(fluid=True)
        for k in want:
            assert np.array_equal(want[k], got[k]), k
        for f in ("fel", "fs", "bin", "bin_off", "rho_s", "rho_bar", "force"):
            assert np.array_equal(a.field(f), w.field(f)), f
    beads, off = a.field("bin_beads"), a.field("bin_off")
    bins = a.field("bin")
    for k in np.nonzero(np.diff(off))[0]:
        assert np.array_equal(np.sort(beads[off[k]:off[k + 1]]), np.nonzero(bins == k)[0])
    ow = O.World(spec)
    st = O.rollout(ow, 12)
    assert_field("disp", a.state()["disp"], t2n(st.D), 1e-5)
    c = World.load(a.save(), spec)
    for w in (a, c):
        w.step(20)
    for k, v in a.state(fluid=True).items():
        assert np.array_equal(v, c.state(fluid=True)[k]), k


@pytest.mark.parametrize("H,W,n_fil", [(32, 96, 110), (64, 64, 64), (96, 128, 700), (256, 256, 4096)])
@pytest.mark.parametrize("sigma", [0.5, 1.0, 2.0])
def test_dense_tiles_deposit(H, W, n_fil, sigma):
    """Tiles of a bead a cell and more, whose fixed-point scale comes from the
    beads' cells (or, with an axis that one tile covers, from a first deposit):
    the density and its filter against the oracle at 1e-6 of their scale (sums
    of 32-bit weights: 2^-24 each, some tens of terms)."""
    rng = np.random.default_rng(n_fil)
    B = 32
    x = np.concatenate([rng.uniform(0, W) + np.arange(B) * 0.9 for _ in range(n_fil)]) % W
    y = np.repeat(rng.uniform(0, H, n_fil), B) + rng.uniform(-0.3, 0.3, n_fil * B)
    x, y = np.mod(x, W).astype(np.float32), np.mod(y, H).astype(np.float32)
    x[x >= W] = 0
    y[y >= H] = 0
    J = n_fil * (B - 2)
    spec = synth._world("dense", H, W, [B] * n_fil, x, y, np.zeros(n_fil * (B - 1), np.float32), np.zeros(J),
                        np.zeros(J), np.zeros(J), np.zeros(J), params=synth.Params(k_rep=1e-3, sigma=sigma))
    ow = O.World(spec)
    _, rec = O.step(ow, ow.initial_state(), record=True)
    w = World(spec)
    w.step(1)
    assert_field("rho_s", w.field("rho_s"), t2n(rec["rho_s"]), 1e-6)
    assert_field("rho_bar", w.field("rho_bar"), t2n(rec["rho_bar"]), 1e-6)
    b = World(spec)
    step_batched([b, World(synth.world_random(4, (40, 72), 5))], 1)
    assert np.array_equal(w.field("rho_s"), b.field("rho_s"))


@pytest.mark.parametrize("H,W,n_fil,sigma", [(32, 96, 40, 1.0), (40, 32, 12, 0.5), (200, 328, 60, 2.0), (256, 256, 2000, 1.0),
                                             (800, 808, 700, 1.0)])
def test_narrow_deposit_blocks(H, W, n_fil, sigma):
    """A world in a batch of many tiles, whose deposit takes blocks of 128
    threads, against the same world alone (wider blocks, but for the last) and
    the persistent step (256 threads): bitwise the same.  Folded axes, ragged
    and dense tiles, empty ones, other filter widths."""
    from paper_2607_02954_gb300 import set_launch_config
    rng = np.random.default_rng(H + W)
    B = 24
    x = np.concatenate([rng.uniform(0, W) + np.arange(B) * 0.9 for _ in range(n_fil)]) % W
    y = np.repeat(rng.uniform(0, H, n_fil), B) + rng.uniform(-0.3, 0.3, n_fil * B)
    x, y = np.mod(x, W).astype(np.float32), np.mod(y, H).astype(np.float32)
    x[x >= W] = 0
    y[y >= H] = 0
    J = n_fil * (B - 2)
    spec = synth._world("narrow", H, W, [B] * n_fil, x, y, np.zeros(n_fil * (B - 1), np.float32), np.zeros(J),
                        np.zeros(J), np.zeros(J), np.zeros(J), params=synth.Params(k_rep=1e-3, sigma=sigma))
    alone, persistent, batched = World(spec), World(spec), World(spec)
    if sigma == 1.0:   # (the persistent step takes a filter half width of 4 only)
        set_launch_config([persistent], persistent=4)
    alone.step(3)
    persistent.step(3)
    sparse = [World(synth.world_random(k, (256, 288), 2)) for k in range(9)]   # 648 tiles
    step_batched([batched] + sparse, 3)
    want = alone.state(fluid=True)
    for w in (persistent, batched):
        for k, v in w.state(fluid=True).items():
            assert np.array_equal(want[k], v), k
        for k in ("rho_s", "rho_bar"):
            assert np.array_equal(alone.field(k), w.field(k)), k


@pytest.mark.parametrize("n", [3, 4])
def test_read_outs_after_a_rewind_and_a_backward(n):
    """The bins of the last step that ran can be read after the counter has
    moved back, whichever parity it had, and after a reverse sweep of one
    segment the fields are the rollout's last step's."""
    spec = crowded(14)
    w = World(spec)
    w.rollout_forward(n, n)
    want = {f: w.field(f) for f in ("bin_off", "rho_s", "rho_bar", "force")}
    gx = torch.ones(spec.N, device="cuda")
    w.rollout_backward(gx, gx)
    for f, v in want.items():
        assert np.array_equal(v, w.field(f)), f
    w.rollout_rewind()
    assert np.array_equal(want["bin_off"], w.field("bin_off"))
    assert np.array_equal(want["rho_s"], w.field("rho_s"))


def room(counts):
    """Slots that bins of these bead counts are given."""
    return (counts + counts // 4 + 16 + 7) // 8 * 8


def uniform_flow(H, W, ux, uy):
    cx = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
    cy = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]
    wt = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    cu = cx * ux + cy * uy
    return np.broadcast_to(wt * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy)), (9, H, W)).astype(np.float32)


def drifting(seed, **kw):
    """A crowd carried across bins by a uniform flow (beads further apart with
    direct forcing, whose passes overshoot where several share a cell)."""
    spec = synth.world_random(seed, (72, 64), 12) if kw.get("ib") else crowded(seed, n_fil=40, at=(20.0, 20.0))
    for k, v in kw.items():
        setattr(spec.params, k, v)
    spec.f0 = uniform_flow(spec.H, spec.W, 0.3, 0.1)
    return spec


def read_outs(w, names=("bin", "bin_off", "rho_s", "rho_bar", "force", "fs", "fel")):
    """The fields of the last step (and the beads of each bin in order)."""
    out = {f: w.field(f) for f in names}
    off, beads = out["bin_off"], w.field("bin_beads")
    out["bin_beads"] = np.concatenate([np.sort(beads[off[k]:off[k + 1]]) for k in range(len(off) - 1)])
    return out


def assert_same(got, want, what):
    for k in got:
        assert np.array_equal(want[k], got[k]), (what, k)


@pytest.mark.parametrize("kw", [{}, dict(layers=2), dict(ib=1, mdf_iters=2)])
@pytest.mark.parametrize("n,every,stored,before", [(3, 3, False, 0), (4, 4, False, 0), (16, 16, False, 0),
                                                   (17, 17, False, 5), (32, 16, False, 0), (32, 32, False, 3),
                                                   (16, 0, True, 0), (17, 0, True, 0), (32, 0, True, 21)])
def test_read_outs_after_rollouts_backwards_and_rewinds(n, every, stored, before, kw):
    """The read-outs are those of the last step that ran: after a recorded or
    stored rollout (also one that ends where a layout of the slots is due),
    after the reverse sweep (whose last re-run is the first segment), after a
    rewind, and in an image saved there."""
    spec = drifting(31, **kw)
    if n >= 16:   # the first and the last step ask for other slots, so a layout between them and the read-out shows
        last = np.diff(O.cell_and_bin(spec.x, spec.y, spec.H, spec.W, 8)[2])
        moved = np.mod(spec.x + 0.3 * (n + before), spec.W), np.mod(spec.y + 0.1 * (n + before), spec.H)
        assert (room(last) != room(np.diff(O.cell_and_bin(*moved, spec.H, spec.W, 8)[2]))).any()
    plain, w = World(spec), World(spec)
    plain.step(before)
    w.step(before)
    first = None
    if not stored and every < n:
        first = World(spec)
        first.step(before + every)
        first = read_outs(first)
    plain.step(n)
    end = read_outs(plain)
    w.rollout_forward(n, every or n, stored=stored)
    assert_same(read_outs(w), end, "forward")
    w.rollout_rewind()
    assert_same(read_outs(w), end, "rewind")
    w.rollout_forward(n, every or n, stored=stored)
    gx = torch.ones(spec.N, device="cuda")
    w.rollout_backward(gx, gx)
    # (what goes through the slots alone: F_el, F_s, the normals that the layer points of two layers need and the
    # total force of direct forcing stay in the re-run's records)
    names = ("bin", "bin_off", "rho_s", "rho_bar") + (() if kw else ("force",))
    want = end if first is None else first
    assert_same(read_outs(w, names), want, "backward")
    w.rollout_rewind()
    assert_same(read_outs(w, names), want, "rewind after backward")
    loaded = World.load(w.save(), spec)
    assert_same(read_outs(loaded, names), want, "load")
    for other in (w, loaded):
        other.step(n)
        assert_same(read_outs(other), end, "again")
        assert_same(other.state(fluid=True), plain.state(fluid=True), "again")


@pytest.mark.parametrize("before", [3, 16, 37])
def test_steps_after_a_run_that_timed_out_stay_in_bounds(before):
    """A persistent run that ends at its first barrier leaves its PBD's counts
    behind, and the layout of a later step gives them slots that hold no
    record.  The world's state is unspecified then, but its steps and read-outs
    stay within their arrays, and other worlds are not affected."""
    from paper_2607_02954_gb300 import _lib, set_launch_config
    lib = _lib.load()
    spec, other = drifting(31), synth.world_random(4, (40, 72), 5)
    w, a, b = World(spec), World(other), World(other)
    w.step(before)
    set_launch_config([w], persistent=4)
    _lib.check(lib.mc_debug_barrier_test(1, 2_000_000))   # 2 ms
    try:
        w.step(1)
        with pytest.raises(_lib.MCError):
            w.check()
    finally:
        _lib.check(lib.mc_debug_barrier_test(0, 1_000_000_000))
    set_launch_config([w], persistent=0)
    _lib.check(lib.mc_world_clear_flags(w.handle, None))
    for _ in range(40):
        step_batched([w, a], 1)
        w.step(1)
        b.step(1)
    got = w.state(fluid=True)
    assert np.isfinite(got["x"]).all() and (got["x"] >= 0).all() and (got["x"] <= spec.W).all()
    for f in ("rho_s", "rho_bar", "force", "bin_off", "bin_beads"):
        w.field(f)
    w.save()
    assert_same(a.state(fluid=True), b.state(fluid=True), "other world")


@pytest.mark.parametrize("kw", [{}, dict(layers=2), dict(ib=1, mdf_iters=1)])
def test_read_outs_before_the_first_step_are_zero(kw):
    """A world that no step has binned yet, in memory that another world's
    records may have left behind, created and loaded."""
    spec = drifting(31, **kw)
    old = World(spec)
    old.step(3)
    torch.cuda.synchronize()
    old.close()
    w = World(spec)
    for v in (w, World.load(w.save(), spec)):
        for f in ("force", "rho_s", "rho_bar", "bin_off"):
            assert not v.field(f).any(), f
        v.step(2)
    assert_same(v.state(fluid=True), w.state(fluid=True), "steps")


@pytest.mark.parametrize("order", [(0, 1, 2, 3, 7, 6), (0, 3, 7, 6), (0, 1, 2, 3, 4, 5, 6)])
def test_read_outs_between_the_stages_of_a_step(order):
    """A read-out between two stages shows the step in progress (its PBD has
    taken the slots over) and does not disturb it."""
    from paper_2607_02954_gb300 import _lib
    lib = _lib.load()
    spec = drifting(31)
    w, ref = World(spec), World(spec)
    names = ("bin_off", "rho_s", "rho_bar", "force")
    for k in range(3):
        ref.step(1)
        want = read_outs(ref, names)
        for stage in order:
            _lib.check(lib.mc_step_stage(w.handle, stage, None))
            for f in names + ("force", "rho_s"):
                assert np.array_equal(w.field(f), want[f]), (k, stage, f)
            assert_same(read_outs(w, names), want, (k, stage))
        assert_same(w.state(fluid=True), ref.state(fluid=True), k)


@pytest.mark.parametrize("at", [(20.2, 20.2), (20.5, 20.5), (20.9, 20.1), (31.4, 9.5)])
@pytest.mark.parametrize("n_fil", [300, 700, 3000, 9000])
def test_a_crowded_spot_leaves_its_tile_the_bits_of_the_largest_sum(at, n_fil):
    """A crowd in a few cells and single beads elsewhere in the tile: the
    deposit's fixed point is as fine as the largest sum M of the tile allows
    (the largest k with M 2^k < 2^30), so a cell that t beads reach is off by
    t halves of 2^-k, and by the rounding of their 32-bit weights (products of
    two factors of at most 1/2, each off by 2^-25: 2^-25 a bead)."""
    H, W, B = 96, 96, 2
    rng = np.random.default_rng(n_fil)
    h = rng.uniform(0, 2 * np.pi, n_fil + 12)
    x0, y0 = (rng.uniform(8, 30, n_fil + 12) for _ in range(2))
    x0[:n_fil] = at[0] + rng.uniform(0, 0.05, n_fil)
    y0[:n_fil] = at[1] + rng.uniform(0, 0.05, n_fil)
    L = np.where(np.arange(n_fil + 12) < n_fil, 0.05, 1.0)
    x = np.stack([x0, x0 + L * np.cos(h)], 1).ravel().astype(np.float32)
    y = np.stack([y0, y0 + L * np.sin(h)], 1).ravel().astype(np.float32)
    e = np.zeros(0)
    spec = synth._world("spot", H, W, [B] * len(h), x, y, h.astype(np.float32), e, e, e, e,
                        params=synth.Params(k_rep=1e-6, kappa=1e-6))
    ow = O.World(spec)
    _, rec = O.step(ow, ow.initial_state(), record=True)
    want = t2n(rec["rho_s"])
    reach = np.zeros((H, W), int)
    for b in range(-1, 3):
        for a in range(-1, 3):
            np.add.at(reach, ((np.floor(y).astype(int) + b) % H, (np.floor(x).astype(int) + a) % W), 1)
    w = World(spec)
    w.step(1)
    got = w.field("rho_s").astype(np.float64)
    checked = 0
    for ty in range(0, H, 32):
        for tx in range(0, W, 32):
            # the tile and what its filter reads
            rows, cols = np.arange(ty - 3, ty + 35) % H, np.arange(tx - 8, tx + 40) % W
            k = 30 - np.frexp(want[np.ix_(rows, cols)].max())[1]
            if k >= 24:
                continue
            t = np.s_[ty:ty + 32, tx:tx + 32]
            few = (reach[t] > 0) & (reach[t] < 8)
            err = np.abs(got[t] - want[t]) / reach[t].clip(min=1)
            assert (err[few] <= 2.0 ** -(k + 1) + 2.0 ** -25).all(), (k, err[few].max() * 2.0 ** (k + 1))
            checked += few.sum()
    assert checked


@pytest.mark.parametrize("n_worlds", [1, 3])
def test_a_long_persistent_run_lays_the_slots_out_again(n_worlds):
    """A band of beads carried out of its bins: one persistent run of 192 steps
    equals twelve of 16 bitwise and takes about their time (every step reading
    all the beads that have left their first bins took several times as long)."""
    from paper_2607_02954_gb300 import set_launch_config
    H, W, B, n_fil = 256 if n_worlds > 1 else 512, 512, 32, 4096
    rng = np.random.default_rng(5)
    x = (np.repeat(rng.uniform(0, 64, n_fil), B) + rng.uniform(0, 0.1, n_fil * B)).astype(np.float32)
    y = np.mod(rng.uniform(0, H, (n_fil, 1)) + np.arange(B), H).astype(np.float32).ravel()
    y[y >= H] = 0
    J = n_fil * (B - 2)
    spec = synth._world("band", H, W, [B] * n_fil, x, y, np.full(n_fil * (B - 1), np.pi / 2, np.float32), np.zeros(J),
                        np.zeros(J), np.zeros(J), np.zeros(J), params=synth.Params(k_rep=1e-4, kappa=1e-3))
    spec.f0 = uniform_flow(H, W, 0.3, 0.0)
    long, short = ([World(spec) for _ in range(n_worlds)] for _ in range(2))
    ms = []
    for ws, runs in ((long, [16, 192]), (short, [16] + [16] * 12)):
        set_launch_config(ws, persistent=4)
        step_batched(ws, runs[0])
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        for n in runs[1:]:
            step_batched(ws, n)
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    print("ms of one run, of twelve:", ms)
    for a, b in zip(long, short):
        a.check()
        assert_same(a.state(fluid=True), b.state(fluid=True), "state")
    assert ms[0] < 1.5 * ms[1], ms


def test_a_captured_step_replays_like_single_steps():
    """One step captured by the caller into a graph of its own and replayed 40
    times (the slots are laid out inside the capture) equals 40 single steps."""
    spec = crowded(19)
    a, b = World(spec), World(spec)
    a.step(1)
    b.step(1)
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        a.step(1, stream=s)
    for _ in range(40):
        g.replay()
        b.step(1)
    torch.cuda.synchronize()
    x, y = a.state_device(), b.state_device()
    for k in x:
        assert torch.equal(x[k], y[k]), k
