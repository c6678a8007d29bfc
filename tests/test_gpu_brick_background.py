"""A brick store whose background colours differ between neighbouring tiles (a
store need not come from ebit_pack_bricks): the edges across those tiles' faces
carry markers, whose offsets the tiles outside the store hold as 0, whatever the
context held before."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_26361_gb300 import ebit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n3", [(16, 24, 32), (41, 18, 33), (9, 65, 16)])
@pytest.mark.parametrize("bricks", [0, 5])
def test_offsets_of_the_tiles_outside_the_store_are_zero(n3, bricks):
    rng = np.random.default_rng(sum(n3) + bricks)
    nx, ny, nz = n3
    td = [-(-n // 8) for n in n3]
    nt = td[0] * td[1] * td[2]
    bricks = min(bricks, nt)
    tiles = np.sort(rng.choice(nt, bricks, replace=False)).astype(np.int32)
    bg = rng.integers(0, 2, nt, dtype=np.uint8)
    bcb = 15 * rng.integers(0, 2, (bricks, 512), dtype=np.uint8)  # (a face of the lowest corner's colour)
    bs = rng.uniform(0.1, 0.9, (bricks, 3, 512))
    # the state it describes
    cb, s = np.empty((nz, ny, nx), np.uint8), np.zeros((3, nz, ny, nx))
    for t in range(nt):
        x, y, z = 8 * (t % td[0]), 8 * (t // td[0] % td[1]), 8 * (t // (td[0] * td[1]))
        sel = (slice(z, min(z + 8, nz)), slice(y, min(y + 8, ny)), slice(x, min(x + 8, nx)))
        cut = tuple(slice(0, q.stop - q.start) for q in sel)
        k = np.searchsorted(tiles, t)
        if k < bricks and tiles[k] == t:
            cb[sel] = bcb[k].reshape(8, 8, 8)[cut]
            for a in range(3):
                s[a][sel] = bs[k, a].reshape(8, 8, 8)[cut]
        else:
            cb[sel] = 15 * bg[t]
    c = cb & 1
    m = np.stack([c != np.roll(c, -1, 2 - a) for a in range(3)])
    s[~m] = 0.0
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    g = ebit.Grid(*n3)
    # every edge of the context holds an offset first, in both buffers
    chess = (np.indices(cb.shape).sum(0) & 1).astype(np.uint8) * 15
    g.set_state(dev(chess), dev(np.full(s.shape, 0.75)))
    g.sweep(0, dev(np.full(cb.shape, 0.1)), 0.1 * g.h)
    g.unpack_bricks({"tiles": dev(tiles), "cb": dev(bcb), "s": dev(bs), "bg": dev(bg)})
    got_cb, got_s = (t.cpu().numpy() for t in g.get_state())
    assert np.array_equal(got_cb, cb) and np.array_equal(got_s, s)
    u = rng.uniform(-0.5, 0.5, cb.shape)
    g.sweep(1, dev(u), 0.9 * g.h)
    o, _ = oracle.sweep(oracle.State(cb, s), 1, u, 0.9)
    got_cb, got_s = (t.cpu().numpy() for t in g.get_state())
    co = o.cb & 1
    mo = np.stack([co != np.roll(co, -1, 2 - a) for a in range(3)])
    assert np.array_equal(got_cb, o.cb) and np.abs(got_s - o.s)[mo].max(initial=0.0) <= 1e-12
    g.close()
