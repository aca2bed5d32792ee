"""The forms in which the one-step kernels read their source (ordered, plain and read-only loads; overlapping and
ordinary launches): the same bits whichever a size, a storage form or a launch shape leads to."""
import numpy as np
import pytest
import torch

from paper_1404_2363_gb300.solver import Solver

pytestmark = pytest.mark.gpu

D2 = [[0.03, 0.005], [0.005, 0.04]]
D3 = [[0.03, 0.005, -0.004], [0.005, 0.025, 0.003], [-0.004, 0.003, 0.035]]


def run(n, storage, u, bc, bc_x, launch, chunks, wait=False):
    lattice = 15 if len(n) == 3 else 9
    g = torch.Generator(device="cuda").manual_seed(11)
    s = Solver(lattice=lattice, nx=n[0], ny=n[1], nz=n[2] if lattice == 15 else 1, storage=storage, bc=bc, bc_x=bc_x,
               phi_w=(0.4, 0.2))
    s.set_D(np.array(D3 if lattice == 15 else D2))
    if launch is not None:
        s.set_launch(*launch)
    sched = torch.rand((5, s.dim), device="cuda", generator=g)
    shape = (s.dim,) + s.shape if u == "field" else (s.dim, n[1])
    if u != "none":
        s.set_velocity(0.04 * torch.rand(shape, device="cuda", generator=g) - 0.02, sched, kind=u)
    s.set_phi(torch.rand(s.shape, device="cuda", generator=g))
    for k in chunks:
        s.step(k)
        if wait:
            torch.cuda.synchronize()
    state = s.get_state()[0].cpu().numpy()
    s.close()
    return state


@pytest.mark.parametrize("n,u,bc_x,launch", [
    ((64, 24, 20), "field", ("bounceback", "noflux"), (256, 1)), ((97, 60), "field", ("noflux", "bounceback"), (256, 1)),
    ((64, 24, 20), "none", ("bounceback", "noflux"), (256, 1)), ((64, 24, 20), "row", ("periodic", "periodic"), (128, 9)),
    ((64, 24, 20), "row", ("periodic", "periodic"), (256, 9)), ((64, 24, 20), "field", ("periodic", "periodic"), (32, 5))])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_overlapping_launches_equal_separate_ones(storage, n, u, bc_x, launch):
    """Many launches in a row on a grid small enough for several to be resident at once, against the same with the
    stream drained after each."""
    if storage == "f32":
        launch = (launch[0], 1)
    a, b = (run(n, storage, u, ("noflux", "bounceback"), bc_x, launch, [1] * 300, wait) for wait in (True, False))
    assert np.array_equal(a, b)
    assert np.array_equal(a, run(n, storage, u, ("noflux", "bounceback"), bc_x, launch, [300]))


def repeated(n, axis, times, storage, u, bc, launch, steps=7):
    """The state of a grid that repeats a small one `times` times along an axis (0: x, 1: y, 2: z), copies first."""
    lattice = 15 if len(n) == 3 else 9
    g = torch.Generator(device="cuda").manual_seed(13)
    dim = len(n)
    k = dim - 1 - axis                                  # array axis
    rep = [1] * dim
    rep[k] = times
    big = [m * (times if d == axis else 1) for d, m in enumerate(n)]
    s = Solver(lattice=lattice, nx=big[0], ny=big[1], nz=big[2] if dim == 3 else 1, storage=storage, bc=(bc, bc))
    s.set_D(np.array(D3 if dim == 3 else D2))
    s.set_launch(*launch)
    shape = tuple(reversed(n))
    phi = torch.rand(shape, device="cuda", generator=g)
    a = 0.04 * torch.rand((dim,) + shape, device="cuda", generator=g) - 0.02
    sched = torch.rand((5, dim), device="cuda", generator=g)
    if u == "field":
        s.set_velocity(a.repeat([1] + rep), sched)
    s.set_phi(phi.repeat(rep))
    s.step(steps)
    state = s.get_state()[0]
    cells, q = s.ncell, 9 if dim == 2 else 15
    s.close()
    elem = 4 if storage == "f32" else 2
    f = state[:cells * q * elem].reshape([q] + list(reversed(big)) + [elem])
    f = f.unflatten(1 + k, (times, n[axis])).movedim(1 + k, 0)
    return f.contiguous()


@pytest.mark.parametrize("storage,n,axis,times,u,bc,launch", [
    ("bf16", (64, 40, 30), 2, 10, "field", "noflux", (32, 5)), ("f16", (64, 40, 30), 2, 10, "field", "bounceback", (64, 5)),
    ("f16", (64, 40, 30), 2, 42, "none", "noflux", (128, 5)), ("bf16", (64, 40, 30), 2, 35, "field", "periodic", (64, 5)),
    ("f16", (64, 40), 0, 850, "field", "noflux", (128, 2)), ("bf16", (64, 40), 0, 3300, "field", "bounceback", (256, 1)),
    # blocks so many that starting them overlapped would take longer than the nodes
    ("f32", (40, 40), 1, 400, "field", "periodic", (64, 1)), ("f32", (40, 40, 20), 2, 30, "none", "periodic", (96, 1)),
    ("f16", (40, 40, 20), 2, 30, "field", "noflux", (64, 1)), ("bf16", (40, 40), 1, 400, "none", "periodic", (64, 2)),
    ("bf16", (40, 40, 20), 2, 30, "none", "noflux", (32, 5))])
def test_large_grids_give_the_bits_of_small_ones(storage, n, axis, times, u, bc, launch):
    """A size from which the launch and the loads take another form, as copies of a grid below it."""
    small = repeated(n, axis, 1, storage, u, bc, launch)
    assert bool((repeated(n, axis, times, storage, u, bc, launch) == small).all())


@pytest.mark.parametrize("launch,steps,launches", [((256, 1), 11, 11), ((128, 11), 11, 4), ((128, 12), 11, None)])
def test_launches_are_counted(launch, steps, launches):
    """One per step, or per group of steps: the walk takes 4 + 4 + 2 + 1; the tiles groups of at most eight."""
    s = Solver(nx=320, ny=200)
    s.set_D(np.array(D2))
    s.set_launch(*launch)
    s.set_phi(torch.rand((200, 320), device="cuda"))
    s.step(steps)
    assert s.launches == launches if launches else 2 <= s.launches < steps
    s.close()
