"""What the autotuner times (host logic, no GPU): the two block sizes of the per-cell
passes on one tile shape, for the trace runs the same blocks whatever the shape."""
import json

from paper_1201_5651_gb300 import autotune, oots


class _Ctx:
    shape, precision = (64, 64, 64), oots.OOTS_MIXED

    def __init__(self):
        self.tiles, self.blocks, self.runs = [], [], 0

    def set_tile_shape(self, s):
        self.tiles.append(s)

    def set_cell_block(self, b):
        self.blocks.append(b)

    def profile_substep(self):
        self.runs += 1
        return [("sweep1", 1.0), ("half", 3.0 if self.blocks[-1:] == [256] else 2.0)]


def test_only_block_sizes_are_timed(tmp_path):
    path = str(tmp_path / "tune.json")
    c = _Ctx()
    assert autotune.tune(c, "GB300", 1, repeats=2, use_cache=False, path=path) == autotune.TILE_SHAPE
    assert c.tiles == [autotune.TILE_SHAPE] and c.blocks == [128, 256, 128]
    assert c.runs == 2 * (1 + 2)
    entry = json.load(open(path))["GB300|mixed|side64|S1|G1"]
    assert (entry["shape"], entry["cell_block"]) == (autotune.TILE_SHAPE, 128)
