"""What a batch keeps on the device: 64 bytes a scenario and bus (phasors and
residuals), as its header says, besides the windows and the scenarios' records.
"""
import pytest

from gridcases import random_grid

pytestmark = pytest.mark.gpu


def test_workspace_per_scenario_and_bus():
    import gc
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    gc.collect()   # nothing of earlier tests is freed meanwhile
    nb, S = 20000, 256
    grid = pf.ybus_build(random_grid(nb, 26400, 9))
    keep = pf.batch_create(grid, 1)   # what any batch holds of the grid's size
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    batch = pf.batch_create(grid, S)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert 64 * S * nb <= used <= 68 * S * nb
    del batch, keep
