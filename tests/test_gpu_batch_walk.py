"""PER_STEP batches that take several steps per launch: when they do, and their bits over ranges of rows."""
import numpy as np
import pytest
import torch

from paper_1404_2363_gb300.batch import Batch, poiseuille_row

pytestmark = pytest.mark.gpu

WALLS = [("noflux", "noflux"), ("periodic", "periodic"), ("bounceback", "noflux"), ("noflux", "bounceback"),
         ("bounceback", "bounceback")]


def channels(n, nx, ny, walls=WALLS[:1], spread=0):
    return [{"nx": nx + spread * i, "ny": ny + (3 * i) % (spread + 1), "bc": walls[i % len(walls)],
             "D": [[0.03, 0.004], [0.004, 0.05]],
             "u_row": poiseuille_row(ny + (3 * i) % (spread + 1), 0.08) if i % 4 else None, "x_ref0": float(nx // 5),
             "x_ref_velocity": 0.05, "model": ("A", "B1", "B3")[i % 3]} for i in range(n)]


# us a step by single steps / by the walk: 7.8 / 10.5, 9.5 / 10.5, 10.4 / 13.0, 12.0 / 13.2, 16.7 / 20.6; then 18.7 / 13.5,
# 33.4 / 19.7, 31.2 / 22.8, 66 / 41
@pytest.mark.parametrize("n,nx,ny,steps", [
    (1, 8192, 64, 1), (4, 1100, 128, 1), (32, 300, 64, 1), (2, 8192, 64, 1), (64, 300, 64, 1), (2, 300, 17, 1),
    (8, 8192, 17, 4), (8, 4097, 64, 4), (2, 8192, 128, 4), (64, 1100, 64, 4)])
def test_walk_only_where_it_pays(n, nx, ny, steps):
    b = Batch(channels(n, nx, ny), mode="per_step")
    assert b.launch_info()[0] == steps
    b.close()


@pytest.mark.parametrize("n,nx,ny,ranges", [(6, 3999, 70, 3), (8, 4000, 101, 3), (4, 4001, 128, 5), (4, 8190, 97, 3)])
def test_walk_over_row_ranges(n, nx, ny, ranges):
    """Channels split into ranges of rows, on every wall pair, odd and even row lengths and heights off the 16-row
    tiles, against the persistent cell tiles (one step at a time): fields and moments bit for bit."""
    chs = channels(n, nx, ny, WALLS, spread=5)
    g = np.random.default_rng(17)
    phis = [(0.05 + g.random((c["ny"], c["nx"]))).astype(np.float32) for c in chs]
    out = []
    for mode in ("persistent", "per_step"):
        b = Batch(chs, mode=mode, graph_steps=16)
        if mode == "per_step":
            assert b.launch_info()[0] == 4 and b.launch_info()[1] >= ranges
        b.set_phi(phis)
        m = b.run(21)
        out.append((m, torch.cat([p.reshape(-1) for p in b.get_phi()])))
        b.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])


def test_launch_steps_can_be_chosen_and_keep_the_bits():
    """PER_STEP with tile_rows 1 and 4 on both sides of the rule, in one handle; the autotuner's choice is one of them."""
    for n, nx, ny, rule in ((4, 1100, 100, 1), (8, 4097, 64, 4)):
        chs = channels(n, nx, ny, WALLS, spread=3)
        g = np.random.default_rng(23)
        phis = [(0.05 + g.random((c["ny"], c["nx"]))).astype(np.float32) for c in chs]
        b = Batch(chs, mode="per_step", graph_steps=16)
        out = {}
        for tile, steps in ((0, rule), (1, 1), (4, 4), (0, rule)):
            b.config("per_step", tile)
            assert b.launch_info()[0] == steps
            b.set_phi(phis)
            m = b.run(21)
            out[tile] = (m, torch.cat([p.reshape(-1) for p in b.get_phi()]))
            assert np.array_equal(m, out[0][0]) and torch.equal(out[tile][1], out[0][1])
        b.set_phi(phis)
        mode, tile = b.autotune(16)
        assert b.launch_info()[0] == ((rule if tile == 0 else tile) if mode == "per_step" else 1)
        m = b.run(21)
        assert mode != "per_step" or np.array_equal(m, out[0][0])
        b.close()


def test_autotune_measures_single_steps_against_the_walk():
    """With the walk as the chosen shape of a batch where it is the slower one, tuning ends with single steps again."""
    b = Batch(channels(1, 8192, 64), mode="per_step", tile_rows=4)
    assert b.launch_info()[0] == 4
    b.set_phi([torch.rand((64, 8192))])
    mode, tile = b.autotune(64)
    assert mode != "per_step" or (tile == 0 and b.launch_info()[0] == 1)
    b.close()


def test_persistent_batches_hold_no_sums_of_the_walk():
    """The walk's column sums (2 x 4 strips of 128 bytes a cell tile) are allocated while PER_STEP uses them."""
    chs = channels(16, 4096, 64)
    torch.cuda.synchronize()
    base = torch.cuda.memory_allocated()
    b = Batch(chs, mode="persistent")
    held = torch.cuda.memory_allocated() - base
    b.config("per_step", 0)
    assert b.launch_info()[0] == 4
    sums = 2 * 4 * 128 * 16 * 128 * 4        # 16 channels of 128 x 4 cell tiles
    assert torch.cuda.memory_allocated() - base >= held + sums
    b.config("persistent", 0)
    assert torch.cuda.memory_allocated() - base == held
    b.close()


def compare(chs, steps, graph_steps, tile, seed=31):
    g = np.random.default_rng(seed)
    phis = [(0.05 + g.random((c["ny"], c["nx"]))).astype(np.float32) for c in chs]
    out = []
    for mode, t in (("persistent", 0), ("per_step", tile)):
        b = Batch(chs, mode=mode, tile_rows=t, graph_steps=graph_steps)
        b.set_phi(phis)
        m = b.run(steps)
        out.append((m, torch.cat([p.reshape(-1) for p in b.get_phi()])))
        b.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])


def test_walk_of_narrow_and_low_channels():
    """The walk on channels narrower than a strip and lower than its halo (chosen: no rule takes it there)."""
    g = np.random.default_rng(37)
    chs = []
    for i in range(40):
        nx, ny = int(g.integers(2, 70)), int(g.integers(3, 40))
        chs += channels(1, nx, ny, [WALLS[i % 5]])
        chs[-1]["x_ref0"] = float(nx // 3)
    compare(chs, 29, 16, 4)


def test_chunks_that_no_graph_replays():
    """50 steps in chunks of 64: single steps in whole chunks, the walk in this one."""
    compare(channels(7, 1436, 62, WALLS, spread=3), 50, 64, 0)
