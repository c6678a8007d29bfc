"""The paths a grid's extents and the arrays' alignment choose, against the
oracle, through the C ABI: row masks of whole, clipped and single tiles, strips
of eight tiles, 16-byte and scalar accesses, state arrays on the device and on
the host.  Colours, statuses, masks and counters are exact; offsets, fractions and
curvature within 1e-12 (the bar of the parity tests)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import amr
from oracle import coupling as CP
from paper_2509_26361_gb300 import ebit

pytestmark = pytest.mark.gpu
TOL = 1e-12
# one tile; a last tile of one cell; row groups of 8 just short of, at and past a
# strip of 64; odd rows; rows past two strips
EXTENTS = [(8, 8, 8), (9, 17, 8), (63, 9, 10), (64, 8, 16), (65, 10, 9), (72, 11, 8), (131, 8, 9)]


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def shifted(a):
    """The same values in device memory that starts off a 16-byte boundary (for
    bytes: off an 8-byte one)."""
    t = torch.empty(a.numel() + 1, dtype=a.dtype, device="cuda")[1:]
    t.copy_(a.reshape(-1))
    return t.view(a.shape)


def random_state(n3, seed, density=0.5):
    """A random colour field in canonical form with random offsets (any colour
    field is a state); a lower density leaves uniform tiles beside mixed ones."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = n3
    cb = rng.integers(0, 16, size=(nz, ny, nx), dtype=np.uint8)
    if density < 0.5:
        cb &= np.uint8(14) | (rng.uniform(size=cb.shape) < density).astype(np.uint8)
        cb[:, :, nx // 2:] &= np.uint8(14)
    s = rng.uniform(0.0, 1.0, size=(3, nz, ny, nx))
    c = cb & 1
    for a in range(3):
        sh = lambda v, b: np.roll(v, -1, axis=2 - b)
        s[a][c == sh(c, a)] = 0.0
        e1, e2 = [b for b in range(3) if b != a]
        c10, c01 = sh(c, e1), sh(c, e2)
        c11 = sh(c10, e2)
        sad = (c == c11) & (c10 == c01) & (c != c10)
        bit = np.where(sad, (cb >> (1 + a)) & 1, c)
        cb = (cb & ~np.uint8(1 << (1 + a))) | (bit.astype(np.uint8) << (1 + a))
    return oracle.State(np.ascontiguousarray(cb), np.ascontiguousarray(s))


def marked(cb):
    c = cb & 1
    return np.stack([c != np.roll(c, -1, 2 - a) for a in range(3)])


@pytest.mark.parametrize("n3,density", [(n3, 0.5) for n3 in EXTENTS] + [((64, 8, 16), 0.03), ((72, 16, 8), 0.03), ((136, 8, 8), 0.03)])
def test_sweeps_fractions_and_masks(n3, density):
    rng = np.random.default_rng(sum(n3))
    st = random_state(n3, 3, density)
    g = ebit.Grid(*n3)
    C = torch.full(g.shape, 7.0, dtype=torch.float64, device="cuda")
    ocnt = np.zeros(5, np.int64)
    for d in range(3):
        u = rng.uniform(-0.9, 0.9, size=st.cb.shape)
        g.set_state(dev(st.cb), dev(st.s))
        g.sweep(d, dev(u), 0.9 * g.h)
        o, c = oracle.sweep(st, d, u, 0.9)
        ocnt += c
        cb, s = (t.cpu().numpy() for t in g.get_state())
        assert np.array_equal(cb, o.cb)
        m = marked(cb)
        assert np.abs(s - o.s)[m].max(initial=0.0) <= TOL and np.all(s[~m] == 0.0)
        # whole-grid fractions and the refinement mask of that state
        g.front2vof(C, ebit.EBIT_FULL)
        oC, _ = oracle.front2vof(o)
        assert np.abs(C.cpu().numpy() - oC).max() <= TOL
        mask, count = g.refine_mask()
        ref = amr.refine_mask(o.cb)
        assert np.array_equal(mask.cpu().numpy().astype(bool), ref) and count == int(ref.sum())
        assert np.array_equal(g.pack_bricks()["tiles"].cpu().numpy(), amr.brick_tiles(o.cb))
    cnt = g.counters()
    assert [cnt[k] for k in ebit.COUNTER_NAMES] == list(ocnt)
    g.close()


@pytest.mark.parametrize("wild", [False, True])
@pytest.mark.parametrize("n3", EXTENTS)
def test_full_curvature_scan(n3, wild):
    """Fractions of random full and empty columns with a few cut cells between
    them, some of whose stencils hold height functions; wild: any C is taken, so
    cells beside the cut ones outside [0, 1], negative zeros and values far below
    the smallest fraction, which the heights sum in FP64."""
    rng = np.random.default_rng(5 + sum(n3))
    nx, ny, nz = n3
    lev = rng.integers(1, 3, size=(nz, ny)) + 0.25 * nx + rng.uniform(size=(nz, ny))
    C = np.clip(lev[:, :, None] - np.arange(nx), 0.0, 1.0)
    if wild:
        near = np.abs(np.arange(nx) - lev[:, :, None]) < 2.5
        odd = rng.choice([1.25, -0.5, -0.0, 1e-300, 0.0, 1.0], size=C.shape)
        C = np.where(near & (rng.uniform(size=C.shape) < 0.1), odd, C)
    okh, ost = oracle.hf_curvature(C)
    g = ebit.Grid(*n3)
    for place in (lambda t: t, shifted):
        Cd = place(dev(C))
        kh = place(torch.full(g.shape, 3.0, dtype=torch.float64, device="cuda"))
        st = place(torch.full(g.shape, 9, dtype=torch.uint8, device="cuda"))
        g.curvature(Cd, kh, st, flags=ebit.EBIT_FULL)
        assert np.array_equal(st.cpu().numpy(), ost)
        assert np.abs(kh.cpu().numpy() - okh).max() <= TOL
    g.close()


@pytest.mark.parametrize("n3", [(8, 8, 8), (9, 8, 10), (34, 9, 8)])
def test_one_fluid_terms_off_16_byte_boundaries(n3):
    rng = np.random.default_rng(9)
    shape = n3[::-1]
    C = rng.choice([0.0, 1.0, 0.3, 0.7], size=shape, p=[0.4, 0.4, 0.1, 0.1])
    kh, st = rng.normal(size=shape), rng.integers(0, 6, size=shape, dtype=np.uint8)
    fl = dict(sigma=0.07, rho1=998.0, rho2=1.2, mu1=1e-3, mu2=1.8e-5)
    ref = CP.properties(C, fl["rho1"], fl["rho2"], fl["mu1"], fl["mu2"])
    g = ebit.Grid(*n3)
    f_ref = CP.csf_force(C, kh, st, g.h, fl["sigma"])
    for place in (lambda t: t, shifted):
        out = tuple(place(torch.full(sh, -1.0, dtype=torch.float64, device="cuda")) for sh in (shape, shape, (3,) + shape))
        rho, mu, f = g.one_fluid(place(dev(C)), dev(kh), dev(st), out=out, **fl)
        assert np.array_equal(rho.cpu().numpy(), ref[0]) and np.array_equal(mu.cpu().numpy(), ref[1])
        assert np.array_equal(f.cpu().numpy(), f_ref)
    g.close()


@pytest.mark.parametrize("n3", [(16, 24, 8), (9, 17, 8), (65, 10, 9)])
def test_state_arrays_on_device_and_host(n3):
    """A state taken in from the device (its markers' offsets only), from device
    memory off any boundary, from the host and from a brick store runs on the
    same, and reads back the same through every kind of array."""
    rng = np.random.default_rng(2)
    st = random_state(n3, 6, 0.05)
    junk = st.s + np.where(marked(st.cb), 0.0, rng.uniform(size=st.s.shape))  # offsets of unmarked edges are ignored
    u = [dev(rng.uniform(-0.8, 0.8, size=st.cb.shape)) for _ in range(3)]
    h = ebit.Grid(*n3)
    h.set_state(dev(st.cb), dev(st.s))
    ends = []
    for how in ("device", "shifted", "host", "bricks"):
        g = ebit.Grid(*n3)
        if how == "bricks":
            g.unpack_bricks(h.pack_bricks())
        elif how == "host":
            g.set_state(torch.from_numpy(st.cb), torch.from_numpy(st.s))
        else:
            cb, s = dev(st.cb), dev(junk if how == "device" else st.s)
            g.set_state(*((shifted(cb), shifted(s)) if how == "shifted" else (cb, s)))
        cb, s = g.get_state()
        assert np.array_equal(cb.cpu().numpy(), st.cb) and np.array_equal(s.cpu().numpy(), st.s)
        for n in range(2):
            g.step(n, u, 0.5 * g.h)
        cb, s = g.get_state()
        hb, hs = torch.empty(g.shape, dtype=torch.uint8), torch.empty((3,) + g.shape, dtype=torch.float64)
        ebit.ebit_get_state(g.ctx, g.N, hb, hs)
        ob, os_ = shifted(torch.zeros_like(cb)), shifted(torch.zeros_like(s))
        ebit.ebit_get_state(g.ctx, g.N, ob, os_)
        assert torch.equal(cb.cpu(), hb) and torch.equal(s.cpu(), hs)
        assert torch.equal(cb, ob) and torch.equal(s, os_)
        ends.append((hb, hs))
        g.close()
    for hb, hs in ends[1:]:
        assert torch.equal(hb, ends[0][0]) and torch.equal(hs, ends[0][1])
    h.close()


def test_batch_after_a_state_change_between_sweeps():
    """Lists of a batch made anew when one instance's state is replaced, whole
    and clipped instances together: every instance as a separate context."""
    sizes = [(16, 16, 16), (24, 8, 16), (17, 9, 12)]
    rng = np.random.default_rng(4)
    b = ebit.Batch(sizes)
    ctx = [ebit.Grid(*n3) for n3 in sizes]
    us = []
    for i, n3 in enumerate(sizes):
        st = random_state(n3, 20 + i)
        us.append(tuple(dev(rng.uniform(-0.8, 0.8, size=n3[::-1])) for _ in range(3)))
        b.instance(i).set_state(dev(st.cb), dev(st.s))
        ctx[i].set_state(dev(st.cb), dev(st.s))
    b.set_velocity(us, [0.5 / n3[0] for n3 in sizes])
    for r in range(3):
        b.run(2 * r, 2, graph=r != 1)
        for i, n3 in enumerate(sizes):
            for k in (2 * r, 2 * r + 1):
                ctx[i].step(k, us[i], 0.5 / n3[0])
            got, ref = b.instance(i).get_state(), ctx[i].get_state()
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), (r, i)
        st = random_state(sizes[r], 40 + r)
        b.instance(r).set_state(dev(st.cb), dev(st.s))
        ctx[r].set_state(dev(st.cb), dev(st.s))
    b.close()
    for g in ctx:
        g.close()


@pytest.mark.parametrize("rows", [1, 127, 128, 129, 300])
def test_gradient_at_the_edges_of_its_tiles(rows):
    """Relative L2 error of each parameter block.  The device rounds the backward
    operands to bf16 (relative error up to 2^-9 each, at most two in a chain and
    one in the product: 6e-3); FP32 sums add far less."""
    from oracle import mlp as omlp

    rng = np.random.default_rng(rows)
    p = (omlp.init_params(3) + rng.normal(scale=0.02, size=omlp.N_PARAMS)).astype(np.float32).astype(np.float64)
    X = omlp.encode(omlp.canonical_stencil(rng.uniform(0, 1, size=(rows, 3, 3, 3))))
    t = rng.uniform(0.05, 0.8, size=rows).astype(np.float32)
    net = ebit.Mlp(p)
    g = net.gradient(dev(X).to(torch.bfloat16), dev(t)).cpu().numpy().astype(np.float64)
    net.close()
    _, ref = omlp.loss_and_grad(p, X, t.astype(np.float64), emulate=True)
    for lo, hi in ((0, 8192), (8192, 8320), (8320, 24704), (24704, 24832), (24832, 24960), (24960, 24961)):
        assert np.linalg.norm(g[lo:hi] - ref[lo:hi]) <= 6e-3 * np.linalg.norm(ref[lo:hi]), (lo, hi)
