"""Sweeps that follow the interface (the band of tiles near markers) on grids
whose last tile of an axis is clipped, small drops that cross the periodic seams
where most tiles are outside the band: against the oracle after every sweep,
against contexts that process every tile, and for batch instances in every tile
shape.  Colours, statuses and counters exact; against the oracle offsets,
fractions and curvature within 1e-12 (the bar of the parity tests), between
paths of the library to the last bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_26361_gb300 import ebit
from paper_2509_26361_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def level_set(n3, drops):
    """max over the drops (centre, radius; cells) of r^2 - |x - c|^2 at the nodes."""
    phi = np.full(n3[::-1], -np.inf)
    for c, r in drops:
        q = 0.0
        for a in range(3):
            d = np.arange(n3[a]) - c[a]
            d -= np.round(d / n3[a]) * n3[a]
            q = q + (d * d).reshape([-1 if 2 - b == a else 1 for b in range(3)])
        phi = np.maximum(phi, r * r - q)
    return phi


def marked(cb):
    c = cb & 1
    return np.stack([c != np.roll(c, -1, 2 - a) for a in range(3)])


# last tiles of 1, 2, 3, 5 and 8 cells, at least four tiles per axis
BOXES = [(25, 26, 27), (34, 25, 32), (29, 27, 33)]
FLOWS = [(1.0, 0.8, 0.9), (-0.9, -1.0, -0.8), (1.0, -0.3, 0.0), (0.0, 0.9, -1.0)]


@pytest.mark.parametrize("v", FLOWS)
@pytest.mark.parametrize("n3", BOXES)
def test_a_drop_over_the_seams_against_the_oracle(n3, v):
    """A drop of radius 2.6 starts two cells before the seams in the direction of
    the flow and is carried some eight cells over them; fractions from what each
    sweep changed."""
    c = [(-4.3 if v[a] > 0 else 4.3) % n3[a] if v[a] else 0.4 for a in range(3)]
    phi = level_set(n3, [(c, 2.6)])
    g = ebit.Grid(*n3)
    g.init(dev(phi))
    st = oracle.init(phi)
    C = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    kh, hs = torch.zeros_like(C), torch.zeros(g.shape, dtype=torch.uint8, device="cuda")
    u = [np.full(st.cb.shape, v[d]) for d in range(3)]
    ud = [dev(x) for x in u]
    cnt = np.zeros(5, np.int64)
    tiles, dt = 0, 0.45 * g.h
    for n in range(18):
        for d in (0, 1, 2) if n % 2 == 0 else (2, 1, 0):
            g.sweep(d, ud[d], dt)
            st, k = oracle.sweep(st, d, u[d], dt / g.h)
            cnt += k
            cb, s = (t.cpu().numpy() for t in g.get_state())
            assert np.array_equal(cb, st.cb), (n, d, np.argwhere(cb != st.cb)[:4])
            m = marked(cb)
            assert np.abs(s - st.s)[m].max() <= TOL and np.all(s[~m] == 0.0), (n, d)
            g.front2vof(C)
            oC, _ = oracle.front2vof(st)
            assert np.abs(C.cpu().numpy() - oC).max() <= TOL, (n, d)
            tiles = max(tiles, g.band_tiles()) if n else tiles
        g.curvature(C, kh, hs)
        okh, ohs = oracle.hf_curvature(oC)
        assert np.array_equal(hs.cpu().numpy(), ohs) and np.abs(kh.cpu().numpy() - okh).max() <= TOL, n
    assert tiles < np.prod([-(-k // 8) for k in n3])  # the band left tiles out
    got = g.counters()
    assert [got[k] for k in ebit.COUNTER_NAMES] == list(cnt)
    g.close()


def drops(rng, n3, count, r0, r1):
    return [(rng.uniform(0.0, 1.0, 3) * n3, rng.uniform(r0, r1)) for _ in range(count)]


def run(n3, phi, u, steps, dense):
    g = ebit.Grid(*n3, dense=dense)
    g.init(dev(phi))
    C = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    kh, hs = torch.zeros_like(C), torch.zeros(g.shape, dtype=torch.uint8, device="cuda")
    for n in range(steps):
        g.step(n, u, 0.6 * g.h)
        g.front2vof(C)
        g.curvature(C, kh, hs)
    out = [*g.get_state(), C, kh, hs]
    cnt = g.counters()
    g.close()
    return out, cnt


def same_events(a, b):
    return {k: v for k, v in a.items() if k != "tiles"} == {k: v for k, v in b.items() if k != "tiles"}


@pytest.mark.parametrize("n3,count", [((97, 75, 61), 5), ((32, 42, 32), 4), ((65, 33, 49), 3), ((50, 41, 26), 2)])
def test_band_equals_every_tile_in_ragged_boxes(n3, count):
    rng = np.random.default_rng(sum(n3))
    phi = level_set(n3, drops(rng, n3, count, 2.0, 5.0))
    u = [dev(a) for a in W.fourier_velocity(n3, rng)]
    (a, ca), (b, cb) = (run(n3, phi, u, 24, dense) for dense in (False, True))
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert same_events(ca, cb) and ca["tiles"] < cb["tiles"]


@pytest.mark.parametrize("shape", [0, 1, 2])
def test_batch_instances_equal_every_tile_in_ragged_boxes(shape):
    rng = np.random.default_rng(7)
    sizes = [(49, 33, 25), (64, 26, 41), (66, 29, 21), (97, 18, 17)]
    b = ebit.Batch(sizes)
    ref, us = [], []
    for i, n3 in enumerate(sizes):
        phi = level_set(n3, drops(rng, n3, 2, 2.0, 3.5))
        u = tuple(dev(a) for a in W.fourier_velocity(n3, rng))
        b.instance(i).init(dev(phi))
        us.append(u)
        ref.append(run(n3, phi, u, 16, True))
    b.set_velocity(us, [0.6 / n3[0] for n3 in sizes])
    b.set_tile_shape(shape)
    Cs = [torch.zeros(n3[::-1], dtype=torch.float64, device="cuda") for n3 in sizes]
    for n in range(0, 16, 2):
        b.run(n, 2, graph=n != 4)
        for i in range(len(sizes)):
            b.instance(i).front2vof(Cs[i])
    b.sync()
    for i, (r, cnt) in enumerate(ref):
        g = b.instance(i)
        cb, s = g.get_state()
        assert torch.equal(cb, r[0]) and torch.equal(s, r[1]) and torch.equal(Cs[i], r[2]), i
        assert same_events(g.counters(), cnt), i
    b.close()
