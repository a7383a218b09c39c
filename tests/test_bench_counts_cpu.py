"""The benchmark's count of the batched kernel's work (no GPU)."""
import bench
from tests.test_plan_source import CSRC


def test_batched_work_is_the_upper_tiles_of_every_round():
    tile_round = 128 * 128 * 64
    assert bench.batched_tile_relaxations([1, 63, 64]) == 0  # one round: no tiles
    assert bench.batched_tile_relaxations([65]) == 2 * 1 * tile_round
    assert bench.batched_tile_relaxations([129]) == 3 * 3 * tile_round
    assert bench.batched_tile_relaxations([1024, 200]) == (16 * 36 + 4 * 3) * tile_round
    # no more than the general mode's grid, and more than the n^3 / 2 relaxations it cannot do without
    for n in (128, 512, 1000, 1500):
        done = bench.batched_tile_relaxations([n])
        assert n ** 3 / 2 < done <= -(-n // 64) * (-(-n // 128)) ** 2 * tile_round


def test_the_kernel_gives_symmetric_graphs_those_tiles():
    src = open(f"{CSRC}/batch.cu").read()
    assert "g.q == 1 ? 0 : g.tiles_x * g.tiles_x" in src
    assert "G[i].tiles = G[i].tiles_x * (G[i].tiles_x + 1) / 2" in src
