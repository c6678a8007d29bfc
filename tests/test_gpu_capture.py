"""Sweeps a caller captures into a CUDA graph of its own: every replay advances
the state that is there when it runs, also where a state was taken in before the
capture or is replaced between replays; compared to the last bit with the same
calls made directly."""
import numpy as np
import pytest
import torch

from paper_2509_26361_gb300 import ebit
from paper_2509_26361_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def problem(n3, seed):
    """A state of spheres (taken from an initialised context) and a velocity field."""
    rng = np.random.default_rng(seed)
    sp = [W.Sphere(tuple(rng.uniform(0.2, 0.8, 3)), rng.uniform(0.12, 0.22)) for _ in range(3)]
    phi, faces = W.sphere_phi_nodes_faces(n3, sp)
    g = ebit.Grid(*n3)
    g.init(dev(phi), dev(faces))
    st = g.get_state()
    g.close()
    return st, tuple(dev(a) for a in W.fourier_velocity(n3, rng))


def direct(n3, st, u, pairs):
    g = ebit.Grid(*n3, dense=True)
    g.set_state(*st)
    for n in range(2 * pairs):
        g.step(n, u, 0.4 * g.h)
    out = g.get_state()
    g.close()
    return out


@pytest.mark.parametrize("within", [False, True])
@pytest.mark.parametrize("dense", [False, True])
def test_steps_captured_after_a_state_was_taken_in(dense, within):
    """The state set on the device before the capture (each replay goes on from
    the one before), or within it (each replay starts from it again)."""
    n3 = (24, 33, 40)
    st, u = problem(n3, 3)
    ref = [direct(n3, st, u, k) for k in (1, 2, 3)]
    side = torch.cuda.Stream()
    g = ebit.Grid(*n3, stream=side, dense=dense)
    g.set_state(*st)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        if within:
            g.set_state(*st)
        g.step(0, u, 0.4 * g.h)
        g.step(1, u, 0.4 * g.h)
    for k in range(3):
        with torch.cuda.stream(side):
            graph.replay()
        torch.cuda.synchronize()
        cb, s = g.get_state()
        want = ref[0 if within else k]
        assert torch.equal(cb, want[0]) and torch.equal(s, want[1]), k
    # and directly again, the state set anew
    g.set_state(*st)
    g.step(0, u, 0.4 * g.h)
    g.step(1, u, 0.4 * g.h)
    cb, s = g.get_state()
    assert torch.equal(cb, ref[0][0]) and torch.equal(s, ref[0][1])
    del graph
    g.close()


def test_batch_sweeps_captured_by_the_caller():
    sizes = [(24, 16, 32), (32, 24, 16)]
    first, second = [problem(n3, 5 + i) for i, n3 in enumerate(sizes)], [problem(n3, 15 + i) for i, n3 in enumerate(sizes)]
    side = torch.cuda.Stream()
    b = ebit.Batch(sizes, stream=side)
    for i in range(2):
        b.instance(i).set_state(*first[i][0])
    b.set_velocity([u for _, u in first], [0.4 / n3[0] for n3 in sizes])
    b.run(0, 2, graph=False)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        for d in (0, 1, 2, 2, 1, 0):
            b.sweep(d)

    def replay(times):
        with torch.cuda.stream(side):
            for _ in range(times):
                graph.replay()
        b.sync()

    replay(2)
    start = [first[0][0], first[1][0]]
    pairs = [3, 3]
    for turn in range(2):
        for i, n3 in enumerate(sizes):
            cb, s = b.instance(i).get_state()
            want = direct(n3, start[i], first[i][1], pairs[i])
            assert torch.equal(cb, want[0]) and torch.equal(s, want[1]), (turn, i)
        if turn == 0:  # one instance's state replaced, the same graph again
            start[1], pairs = second[1][0], [4, 1]
            b.instance(1).set_state(*start[1])
            torch.cuda.synchronize()
            replay(1)
    # and directly from there
    b.run(0, 2, graph=False)
    b.sync()
    for i, n3 in enumerate(sizes):
        cb, s = b.instance(i).get_state()
        want = direct(n3, start[i], first[i][1], pairs[i] + 1)
        assert torch.equal(cb, want[0]) and torch.equal(s, want[1]), i
    del graph
    b.close()


@pytest.mark.parametrize("flags", [ebit.EBIT_FULL, ebit.EBIT_INCREMENTAL])
@pytest.mark.parametrize("density", [0.02, 0.5])
def test_fractions_and_curvature_captured_once(density, flags):
    """One Front2VOF and one curvature call in a graph, replayed: the lists of cut
    and interface cells are the replay's own (with random colours nearly every cell
    is cut, so that two replays' cells would not fit them)."""
    n3 = (24, 16, 40)
    rng = np.random.default_rng(2)
    c = (rng.uniform(size=n3[::-1]) < density).astype(np.uint8)
    cb, s = dev(15 * c), dev(rng.uniform(size=(3,) + c.shape))
    u = tuple(dev(a) for a in W.fourier_velocity(n3, rng))

    def arrays():
        C = torch.zeros(c.shape, dtype=torch.float64, device="cuda")
        return C, torch.zeros_like(C), torch.zeros(c.shape, dtype=torch.uint8, device="cuda")

    d = ebit.Grid(*n3)
    d.set_state(cb, s)
    want, refs = arrays(), []
    for k in range(5):
        d.step(0, u, 0.2 * d.h)
        d.step(1, u, 0.2 * d.h)
        d.front2vof(want[0], ebit.EBIT_FULL)
        d.curvature(*want, flags=ebit.EBIT_FULL)
        refs.append([t.clone() for t in want])
    side = torch.cuda.Stream()
    g = ebit.Grid(*n3, stream=side)
    g.set_state(cb, s)
    out = arrays()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        g.step(0, u, 0.2 * g.h)
        g.step(1, u, 0.2 * g.h)
        g.front2vof(out[0])
        g.curvature(*out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        g.step(0, u, 0.2 * g.h)
        g.step(1, u, 0.2 * g.h)
        g.front2vof(out[0], flags)
        g.curvature(*out, flags=ebit.EBIT_FULL)
    for k in range(5):
        if k in (1, 2, 3):
            with torch.cuda.stream(side):
                graph.replay()
        elif k == 4:  # and directly again
            g.step(0, u, 0.2 * g.h)
            g.step(1, u, 0.2 * g.h)
            g.front2vof(out[0])
            g.curvature(*out)
        torch.cuda.synchronize()
        for a, b in zip(out, refs[k]):
            assert torch.equal(a, b), k
    del graph
    d.close()
    g.close()
