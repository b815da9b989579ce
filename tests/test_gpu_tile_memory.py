"""The shared memory that a tile needs sets which tiles an SM takes: the sizes that the host states when it refuses one."""
import re

import pytest
import torch

from paper_1702_01770_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,tile,need", [(64, (1, 128), 343136), (32, (1, 256), 375904)])
def test_shared_memory_of_tiles(bits, tile, need):
    """Four system types (eight chains and 72 monomers at the most, 3200 bins): the descriptor, the bins and the walkers' slots."""
    from paper_1702_01770_gb300 import phast
    c = phast.Context(inputs.config2(9), pair_precision=bits)
    c.set_tile(*tile)
    with pytest.raises(phast.PhastError, match="shared memory") as e:
        c.sweep(1, c.lnW_zeros())
    torch.cuda.synchronize()
    assert int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)) <= need
    c.close()
