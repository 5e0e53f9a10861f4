"""Source rules of the solve-phase kernels' loads (CPU).

A solve-phase kernel may be launched while its predecessor still writes the
vectors it reads (programmatic dependent launch), so only matrix data, which
the setup alone writes, may go through the non-coherent loads (__ldg, ld_pin)
or be loaded before the wait; a stale vector would give a wrong result without
any error, and only on some schedules, so the rule is checked in the source.
"""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1605_01522_gb300", "csrc", "kernels.cu")
# row pointers and offsets, columns, values, diagonal inverse, rows of the coarse inverse; p, q: the block
# pointer inside the block loaders themselves
MATRIX = {"rp", "sp", "rl", "col", "cp", "val", "v", "vp", "a.dinv", "a", "ar", "p", "q"}


def _source():
    with open(SRC) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_noncoherent_loads_read_matrix_data_only():
    args = re.findall(r"(?:__ldg|ld_pin|ldg_block<[^>]*>|ld_pin_block<[^>]*>)\((?!const)\s*([\w.]+)", _source())
    assert len(args) > 20
    assert set(args) <= MATRIX, sorted(set(args) - MATRIX)


def test_functions_that_wait_take_vectors_without_restrict():
    heads = re.findall(r"void (\w+)\(([^{;]*?\bW wait\b[^{;]*)\)\s*\{", _source())
    names = {n for n, _ in heads}
    assert {"bsr_row", "sell_split_row"} <= names
    for name, params in heads:
        assert not re.search(r"__restrict__ (?:x|b|y|z|d|xout)\b", params), name
