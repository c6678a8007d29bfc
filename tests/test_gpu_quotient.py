"""The quotients of the coupling terms by a known reciprocal equal IEEE division,
on both sides of the operand limits where the division itself is taken (2^-400 and
2^401), for zeros, subnormals and overflow.  On the x-faces of cells 0, 1, 0, 1, ...
with one valid curvature per face the force is ((kappa h / h) (+-1)) / h exactly."""
import numpy as np
import pytest
import torch

from paper_2509_26361_gb300 import ebit

pytestmark = pytest.mark.gpu
N3 = (64, 16, 16)


@pytest.mark.parametrize("h", [1.0 / 48.0, 0.1, 3.0, np.nextafter(2.0, 1.0), 1.0 + 2.0 ** -52, 7e-120, 2.0 ** -400, 2.0 ** -401,
                               np.nextafter(2.0 ** -400, 0.0), 2.0 ** 400 * 1.7, 2.0 ** 401, 1e-300, 1.7e300])
@pytest.mark.parametrize("place", [0, 1])
def test_face_force_is_the_ieee_quotient(h, place):
    rng = np.random.default_rng(11)
    shape = N3[::-1]
    x = np.arange(N3[0]) & 1
    C = np.broadcast_to(x.astype(np.float64), shape).copy()
    st = np.broadcast_to(np.where(x == 1, 1, 0).astype(np.uint8), shape).copy()
    e = rng.integers(-1074, 1024, shape)
    e[::2] = rng.integers(-60, 60, e[::2].shape)
    kh = np.ldexp(rng.uniform(1.0, 2.0, shape), e) * rng.choice([-1.0, 1.0], shape)
    kh[..., 1:24:2] = rng.choice([0.0, -0.0, 2.0 ** -400, np.nextafter(2.0 ** -400, 0.0), 2.0 ** 401,
                                  np.nextafter(2.0 ** 401, 0.0), 5e-324, -1.7e308, np.inf], kh[..., 1:24:2].shape)
    kh[..., 25:40:2] = h * np.nextafter(rng.uniform(1.0, 2.0, kh[..., 25:40:2].shape), 2.0)  # quotients near h's own fraction
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        k = np.where(st == 1, kh, np.roll(kh, 1, 2)) / h  # the valid cell of each x-face
        want = (k * (C - np.roll(C, 1, 2))) / h
    pad = lambda a: torch.cat([torch.zeros(place, dtype=a.dtype), a.reshape(-1)]).cuda()[place:].view(a.shape)
    g = ebit.Grid(*N3, h=float(h))
    Cd, kd = pad(torch.from_numpy(C)), pad(torch.from_numpy(kh))
    out = tuple(torch.full(s, 5.0, dtype=torch.float64, device="cuda") for s in (shape, shape, (3,) + shape))
    _, _, f = g.one_fluid(Cd, kd, torch.from_numpy(st).cuda(), sigma=1.0, rho1=1.0, rho2=1.0, mu1=1.0, mu2=1.0, out=out)
    f = f.cpu().numpy()
    assert np.array_equal(f[0].view(np.int64), want.view(np.int64)), np.argwhere(f[0] != want)[:4]
    assert not f[1:].any()
    g.close()
