"""bench.py counts transform work at the padded lengths the library reports, not at a rule of its own (no GPU)."""
import types

import bench


class _Context:
    def launch_config(self, i):
        return {"Px": (80, 224)[i], "Py": (96, 64)[i]}


def _workload():
    strings = [types.SimpleNamespace(nx=40, ny=45, nz=2), types.SimpleNamespace(nx=100, ny=30, nz=3)]
    return types.SimpleNamespace(strings=strings)


def test_lengths_come_from_the_context():
    assert bench.group_lengths(_Context(), _workload()) == {(40, 45, 2): (80, 96), (100, 30, 3): (224, 64)}


def test_flop_count_takes_them():
    # 2 pairs x (2 x 80 kx x 6 lines x 5 x 64 x 6 + 80 x 64 x 36 x 4): lengths 80 and 64 for 40 and 32 sites
    assert bench.yz_flops_group(40, 32, 2, 4, (80, 64)) == 2 * (2 * 80 * 6 * 5 * 64 * 6 + 80 * 64 * 36 * 4)
    assert bench.yz_flops_group(40, 32, 2, 4) != bench.yz_flops_group(40, 32, 2, 4, (96, 64))
