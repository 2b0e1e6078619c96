"""Marshalling of a step's row arrays (binding.make_step), on the CPU: what the packed block holds, and the
inputs it does not take, which go through int() one by one."""
import numpy as np
import pytest

from paper_2512_03416_b200 import binding as B


def rows_of(st):
    return [[getattr(st, f)[i] for i in range(st.n_rows)] for f in ("slot", "q_len", "ctx_len")]


@pytest.mark.parametrize("n", [0, 1, 4, 203])
@pytest.mark.parametrize("kind", [list, tuple, lambda v: np.array(v, dtype=np.int64), lambda v: [float(x) for x in v]],
                         ids=["list", "tuple", "numpy", "floats"])
def test_a_step_holds_its_rows_and_addresses(n, kind):
    want = [list(range(n)), [1 + i % 7 for i in range(n)], [1000 * i for i in range(n)]]
    st, _keep = B.make_step(*[kind(v) for v in want], 0x10, (1 << 63) + 16, 0, 0x40, 3)
    assert (st.n_rows, st.flags, st.q, st.k_new, st.v_new, st.out) == (n, 3, 0x10, (1 << 63) + 16, None, 0x40)
    assert rows_of(st) == want


def test_a_step_outlives_its_second_result():
    steps = [B.make_step([i], [i + 1], [i + 2])[0] for i in range(200)]
    assert all(rows_of(st) == [[i], [i + 1], [i + 2]] for i, st in enumerate(steps))


def test_rows_of_unequal_length_are_not_mixed_up():
    """The first array says how many rows there are: an array with more is refused, one with fewer is zero
    from there on, and no number moves into another array or row."""
    with pytest.raises(IndexError):
        B.make_step([1, 2], [3, 4, 5], [6])          # six numbers for two rows all the same
    assert rows_of(B.make_step([1, 2], [3, 4], [6])[0]) == [[1, 2], [3, 4], [6, 0]]
    assert rows_of(B.make_step([1, 2], [3], [5, 6])[0]) == [[1, 2], [3, 0], [5, 6]]


def test_values_beyond_32_bits_keep_their_low_bits():
    assert rows_of(B.make_step([(1 << 32) + 7, 1], [1, 2], [-(1 << 31) - 1, 4])[0]) == [[7, 1], [1, 2], [(1 << 31) - 1, 4]]
