"""CPU checks of the comparison that decides whether a decode kernel keeps the schedule it worked out ahead of time.

The schedule is made of lengths that a kernel in front may be writing meanwhile: each item of a sequence (a block of its query
rows) loads the length for itself and may find the old one or the new one."""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2509_25224_b200", "csrc")


@pytest.fixture(scope="module")
def item_is_stale(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "libplan.so")
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-I", CSRC, "-Xcompiler", "-fPIC", "-shared",
                           os.path.join(HERE, "plan_check.cu"), "-o", so])
    f = ctypes.CDLL(so).item_is_stale
    ptr = np.ctypeslib.ndpointer(np.int32, flags="C")
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ptr, ctypes.c_void_p, ptr, ctypes.c_int, ctypes.c_int]
    return f


def _prefix(per_item, tile_keys, ovh):
    """Schedule prefix of items with these lengths."""
    tiles = [-(-n // tile_keys) for n in per_item]
    return np.concatenate([[0], np.cumsum([t + (ovh if it else 0) if t else 0 for it, t in enumerate(tiles)])]).astype(np.int32)


def _stale(f, nrb, tile_keys, ovh, per_item, lens, now, first=(0, 0, 0, 0)):
    prefix, first = _prefix(per_item, tile_keys, ovh), np.array(first, np.int32)
    held = None if lens is None else np.array(lens, np.int32)
    return any(f(nrb, tile_keys, ovh, prefix, None if held is None else held.ctypes.data, first, it, int(now[it // nrb])) for it in range(len(per_item)))


@pytest.mark.parametrize("tile_keys,ovh", [(64, 3), (64, 6), (128, 5)])
@pytest.mark.parametrize("nrb", [1, 2, 3])
def test_a_guess_of_old_and_new_lengths_is_found(item_is_stale, nrb, tile_keys, ovh):
    old, new = [100, 1500, 0], [2000, 1500, 700]
    for seen in itertools.product([0, 1], repeat=2 * nrb):            # what the items of the first and the last sequence found
        per_item = [(old, new)[s][0] for s in seen[:nrb]] + [1500] * nrb + [(old, new)[s][2] for s in seen[nrb:]]
        found = [set(per_item[b * nrb:(b + 1) * nrb]) for b in range(3)]
        for lens in itertools.product(*found):                        # any of a sequence's items may have been the last to leave its length
            assert _stale(item_is_stale, nrb, tile_keys, ovh, per_item, lens, new) == (not all(seen)), (seen, lens)


@pytest.mark.parametrize("tile_keys,ovh", [(64, 6), (128, 5)])
def test_a_length_that_changes_no_tile_is_found_on_chip(item_is_stale, tile_keys, ovh):
    for nrb in (1, 2):
        assert _stale(item_is_stale, nrb, tile_keys, ovh, [65] * nrb + [130] * nrb, [65, 130], [66, 130])
        assert not _stale(item_is_stale, nrb, tile_keys, ovh, [65] * nrb + [130] * nrb, [65, 130], [65, 130])


def test_a_part_without_a_unit_keeps_a_right_schedule(item_is_stale):
    # the prefix alone is on chip: the length that the part's first unit was given is looked at, if it has one
    lens = [300, 0, 700]
    for nrb in (1, 2):
        per_item = np.repeat(lens, nrb).tolist()
        assert not _stale(item_is_stale, nrb, 128, 5, per_item, None, lens)
        for it in (0, 2 * nrb):
            assert not _stale(item_is_stale, nrb, 128, 5, per_item, None, lens, (it, 0, 2, lens[it // nrb]))
            assert _stale(item_is_stale, nrb, 128, 5, per_item, None, lens, (it, 0, 2, lens[it // nrb] - 1))
        assert _stale(item_is_stale, nrb, 128, 5, per_item, None, [300, 0, 900])
