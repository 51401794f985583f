"""The host side of a forest handle: the flat parent array that lantern_forest_create_in reads."""
import numpy as np
import pytest

from paper_2502_06352_b200 import binding


def _want(parents, n_nodes, width):
    flat = []
    for b, n in enumerate(n_nodes):
        row = [int(x) for x in parents[b][:n]]
        flat += row + [-1] * (width - len(row))
    return flat


@pytest.mark.parametrize("form", ["lists", "ragged", "tuples", "numpy", "numpy_int64", "floats", "numpy_rows", "tensor"])
def test_flat_parents_of_every_form(form):
    import torch
    rows = [[-1, 0, 0, 1], [-1, 0, 7, 9], [-1, 5, 5, 5], [-1, 0, 1, 2]]
    n_nodes, width = [4, 2, 1, 3], 4
    if form == "lists":
        parents = rows
    elif form == "ragged":
        parents = [r[:n] for r, n in zip(rows, n_nodes)]
    elif form == "tuples":
        parents = tuple(tuple(r) for r in rows)
    elif form == "numpy":
        parents = np.array(rows, dtype=np.int32)
    elif form == "numpy_int64":
        parents = np.array(rows, dtype=np.int64)
    elif form == "floats":
        parents = [[float(x) for x in r] for r in rows]
    elif form == "numpy_rows":
        parents = [np.array(r) for r in rows]
    else:
        parents = torch.tensor(rows)
    assert list(binding._flat_parents(parents, n_nodes, width)) == _want(parents, n_nodes, width)


def test_flat_parents_of_odd_counts():
    rows = [[-1, 0, 0], [-1, 0, 1]]
    for n_nodes in ([0, 3], [3, 5], [-1, 2]):       # refused by the library later, never misread here
        assert list(binding._flat_parents(rows, n_nodes, 3)) == _want(rows, n_nodes, 3)
    assert list(binding._flat_parents([[-1, 0, 0, 0], [-1, 0, 1, 1]], [3, 3], 3)) == [-1, 0, 0, -1, 0, 1]
    big = [[-1, 2 ** 31, 0], [-1, 0, 1]]             # wraps like a C integer, as ctypes does
    assert len(list(binding._flat_parents(big, [3, 3], 3))) == 6


def test_a_forest_of_refused_arguments_says_so_before_any_device_memory_is_asked_for():
    """Sizes the library refuses and trees that are none: LanternError with the library's status, on a host without a
    GPU too, and no request for an absurd amount of device memory."""
    import torch
    from paper_2502_06352_b200 import Forest, LanternError
    assert binding.lib.lantern_forest_block(2, 60) == 3 * 2 * 60 * 4
    assert binding.lib.lantern_forest_block(1, 1025) == 0 and binding.lib.lantern_forest_block(1 << 22, 1000) == 0
    unsupported, invalid = 2, 1
    for parents, n_nodes, width, status in ([[[-1]], [1], 1025, unsupported], [[[-1, 0, 1, 0]], [4], 4, invalid],
                                            [[[-1, 0]], [3], 3, invalid], [[], [], 4, invalid]):
        with pytest.raises(LanternError) as e:
            Forest(parents, n_nodes, width)
        assert e.value.status == status, (n_nodes, width)
    if not torch.cuda.is_available():
        with pytest.raises(LanternError) as e:           # nothing wrong with the tree: the host has no GPU
            Forest([[-1, 0, 0]], [3])
        assert e.value.status == 4


def test_the_package_imports_without_torchs_private_device_functions():
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import torch\n"
            "for n in ('_cuda_getDevice', '_cuda_getCurrentRawStream'):\n"
            "    if hasattr(torch._C, n): delattr(torch._C, n)\n"
            "class S: cuda_stream = 7\n"
            "torch.cuda.current_device = lambda: 3\n"
            "torch.cuda.current_stream = lambda dev: S\n"
            "import paper_2502_06352_b200.binding as b\n"
            "assert b._current_device() == 3 and b._raw_stream(3) == 7\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=root, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
