"""FP64 -> FP32 on the integer units: every NaN, whatever its payload and sign,
and both infinities become an infinity of that sign (so that a poisoned metric
is seen and not a finite 0), also where the rounding increment would carry out
of the exponent."""
import numpy as np

from test_fp_convert import run


def test_nans_become_infinities(tmp_path):
    rng = np.random.default_rng(1)
    bits = [0x7fffffffffffffff, 0x7ffffffff0000000, 0x7fffffffefffffff, 0x7ff8000000000000, 0x7ff0000000000001,
            0x7ff0000000000000, 0x7fffffff00000000, 0x7ff000000fffffff, 0x7ff0000010000000]
    bits += [0x7ff0000000000000 | int(b) for b in rng.integers(1, 1 << 52, 2000)]
    bits += [0x7fffffff00000000 | int(b) for b in rng.integers(0, 1 << 32, 2000)]
    u = np.array(bits + [b | 1 << 63 for b in bits], dtype=np.uint64)
    got, _ = run(u.view(np.float64), tmp_path)
    assert np.all(np.isinf(got)) and np.array_equal(np.signbit(got), u >> np.uint64(63) == 1)
