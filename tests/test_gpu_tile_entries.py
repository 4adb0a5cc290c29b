"""Which 2D stage kernel a tuning-table entry launches, read from the launched kernels' names: an
entry with a width runs in that width (rows and bands -1: the default band and row geometry of the
width), and no entry, or the autotuner's {0, 0, 96}, runs in the tile chosen for the grid.  On
188 x 70 cells that tile has 32 columns in both precisions, so a stored width that were taken for
"the default" would show."""
import re

import numpy as np
import pytest

from paper_2402_03074_gb300 import _binding as H
from gpu_helpers import gpu_problems_stage

pytestmark = pytest.mark.gpu
NX, NY = 188, 70


def _launched_width(mixed):
    """Columns of the stage kernel that one stage of characteristic Euler launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):  # a process's first recording may start after the launch
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            gpu_problems_stage(NX, NY, 1, mixed, seed=2)
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "stage2d_kernel" in e.name]
        if names:
            break
    else:
        pytest.skip("the profiler records no kernels here")
    assert len(names) == 1, names
    return int(re.search(r"(double|float), (?:\(int\))?(\d+)>", names[0]).group(2))


@pytest.mark.parametrize("mixed", [0, 1])
def test_a_stored_width_is_the_launched_width(tmp_path, mixed):
    import torch
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    path = str(tmp_path / "t.txt")

    def entry(rows, bands, width):
        with open(path, "w") as f:
            f.write(f"{name} 2 1 {mixed} {NX} {NY} {rows} {bands} {width} 0\n")
        assert H.hweno_tuning_load(path) == 1

    try:
        entry(0, 0, 0)
        assert _launched_width(mixed) == 32
        ref = gpu_problems_stage(NX, NY, 1, mixed, seed=2)
        for width in (32, 64, 96, 128, 192):
            entry(-1, -1, width)
            assert _launched_width(mixed) == width
            np.testing.assert_array_equal(gpu_problems_stage(NX, NY, 1, mixed, seed=2), ref)
        entry(0, 0, 96)
        assert _launched_width(mixed) == 32
    finally:
        entry(0, 0, 0)
