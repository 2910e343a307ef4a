"""The background field's per-cell table is a help, not a need: a handle for which the
device has no room beside it is made and steps, with the same bits as one that has a
table; a later allocation of the handle takes the table's room if it has to; a
uniform field has none."""
import gc

import numpy as np
import pytest

from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = (12, 12, 12)  # 1,728 blocks: a table of 25 (mixed) or 50 MB, far above the allocator's 2 MB pages
NB = 1728
B0 = {W.B0_DIPOLE: np.array([0.02, 0.01, 0.05] + [0.0] * 9),
      W.B0_LINEAR: np.array([0.1, 0.2, 0.3, 0.1, 0.02, 0.0, 0.03, -0.1, 0.0, 0.0, 0.01, 0.05]),
      W.B0_UNIFORM: np.array([0.1, 0.2, 0.3] + [0.0] * 9), W.B0_NONE: np.zeros(12)}


def _grid(b0, powell=1):
    q = W.Problem("table", (0.5,) * 3, (2.5,) * 3, ROOT, W.as_leaf_array(W.uniform_leaves(ROOT)), (W.BC_OUTFLOW,) * 6,
                  b0=b0, b0_param=B0[b0], powell=powell)
    x = W.cell_centres(q.lo, q.hi, ROOT, q.leaves)
    s = [np.sin(np.pi * (a + 0.1 * k)) for k, a in enumerate(x)]
    return W.with_state(q, [1 + 0.3 * s[0] * s[1], 0.5 * s[1], 0.4 * s[2], 0.3 * s[0], 0.5 * s[2], 0.4 * s[0],
                            0.6 + 0.2 * s[1], 1 + 0.3 * s[2]])


def _free():
    import torch
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _fill(leave):
    """All but `leave` bytes of the device's free memory."""
    import torch
    return torch.empty(_free() - leave, dtype=torch.uint8, device="cuda")


def _table_bytes(precision):
    return NB * 7 * 512 * (4 if precision == bats.BATS_MIXED else 8)


def _run(q, precision, mlp=None, before_mlp=None):
    with bats.Solver(q, precision=precision) as s:
        used = _free()
        hold = before_mlp() if before_mlp else None
        if mlp is not None:
            s.set_mlp(mlp)
        s.set_state(0, q.U0)
        s.step(3, 0.3)
        U = s.get_state(0)
        del hold
    _free()
    return U, used


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
@pytest.mark.parametrize("b0", [W.B0_DIPOLE, W.B0_LINEAR])
def test_no_room_for_the_table(b0, precision):
    q = _grid(b0)
    _run(q, precision)  # the kernels are loaded
    before = _free()
    U, after = _run(q, precision)
    need = before - after
    assert need >= NB * 8 * 512 * 16 + _table_bytes(precision)
    hold = _fill(need - _table_bytes(precision) // 2)
    V, _ = _run(q, precision)
    del hold
    _free()  # (torch keeps freed memory otherwise)
    assert np.array_equal(U, V)


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
def test_a_later_allocation_takes_the_tables_room(precision):
    q = _grid(W.B0_DIPOLE)
    mlp = np.random.default_rng(3).normal(0, 0.05, size=bats.BATS_MLP_NPARAM).astype(np.float32)
    U, _ = _run(q, precision, mlp)
    # the face inputs and outputs of the network: 3 x 576 faces of 96 + 32 bytes a block
    need = NB * 3 * 576 * 128
    V, _ = _run(q, precision, mlp, lambda: _fill(need - _table_bytes(precision) // 2))
    assert np.array_equal(U, V)


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
def test_a_uniform_field_has_no_table(precision):
    used = []
    for b0 in (W.B0_NONE, W.B0_UNIFORM):
        q = _grid(b0)
        _run(q, precision)
        before = _free()
        used.append(before - _run(q, precision)[1])
    assert used[1] - used[0] < _table_bytes(precision) // 2
