"""Device memory per particle slot, so that a discharge that fits goes on fitting."""
import gc

import pytest

from paper_0705_0497_gb300 import api, inputs

pytestmark = pytest.mark.gpu

CAP = 1 << 26
SLACK = 1.0        # B per slot: tables of fixed size and the allocator's granularity (64 MB)


def _used(torch):
    gc.collect()
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def _config():
    return inputs.base_config(L=0.02, n_cells=128, U=50.0, p=10.0, C_meta=0.0, ion_subcycle=1, weight=1e9, seed=4)


# Two sets of six 4-byte words and 32 B of collision records per slot; 48 B of
# staged births per electron, 16 B per O-.
@pytest.mark.parametrize("species,expected", [(0, 48 + 32 + 48), (1, 48 + 32 + 16), (2, 48 + 32)])
def test_bytes_per_slot(torch_cuda, species, expected):
    cap = [64, 64, 64]
    cap[species] = CAP
    before = _used(torch_cuda)
    d = api.Discharge(_config(), cap)
    per_slot = (_used(torch_cuda) - before) / CAP
    d.close()
    assert per_slot <= expected + SLACK


# The cell sort of the Coulomb collisions: 4 B per cell and tile of 8192 slots.
@pytest.mark.parametrize("species", [0, 1, 2])
def test_bytes_per_slot_of_coulomb(torch_cuda, species):
    cap = [64, 64, 64]
    cap[species] = CAP
    d = api.Discharge(_config(), cap)
    before = _used(torch_cuda)
    d.set_coulomb(63)
    per_slot = (_used(torch_cuda) - before) / CAP
    d.close()
    assert per_slot <= 4 * 128 / 8192 + SLACK


# A network that only runs forward holds its activations, no gradients.
def test_bytes_per_row_of_forward(torch_cuda):
    torch = torch_cuda
    widths, rows = [4] + 14 * [512] + [8], 100_000
    m = api.MLP(widths, seed=1)
    X = torch.zeros(rows, 4, device="cuda")
    torch.cuda.empty_cache()
    before = _used(torch)
    Y = m.forward(X)
    torch.cuda.synchronize()
    per_row = (_used(torch) - before) / rows
    assert Y.shape == (rows, 8)
    # 2 MB granularity of 14 arrays, and of the output's allocator
    assert per_row <= 4 * (14 * 512 + 8) + 15 * 2 ** 21 / rows + 2 ** 21 / rows
    g, _ = m.gradients(X, Y + 1.0)
    assert torch.isfinite(g).all()
    m.close()
