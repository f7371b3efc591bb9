"""The forward tests whose sizes lie within the one launch without a sweep, by
the sweep that the default rule picks there."""
import inspect

import pytest

import test_gpu_forward as forward
from test_gpu_forward import idw  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

RAGGED = [(1, 1), (2, 3), (3, 31), (31, 257), (255, 2047), (256, 2048), (257, 2049), (1000, 4099),
          (4097, 333)]
CASES = ([(forward.test_ragged_sizes, (n, m, p)) for n, m in RAGGED for p in (2.0, 3.0, 3.5)]
         + [(forward.test_general_power, (p,)) for p in (0.5, 1.5, 2.5, 3.5)]
         + [(forward.test_extreme_powers, (0.01,))]
         + [(forward.test_coordinate_ranges, c) for c in
            ((0.0, 1e-20), (1e6, 1000.0), (-3e4, 1e-3), (0.0, 1e12), (5e-3, 1e-6))]
         + [(f, ()) for f in (forward.test_single_point_and_empty_queries,
                              forward.test_near_coincident_takes_fp64_path,
                              forward.test_fp32_overflow_takes_fp64_path,
                              forward.test_permutation_and_constant_field)])


@pytest.mark.parametrize("test,args", CASES,
                         ids=[f"{t.__name__[5:]}-{'-'.join(map(str, a))}" for t, a in CASES])
def test_by_a_sweep(test, args, idw, swept):  # noqa: F811
    assert len(inspect.signature(test).parameters) == 1 + len(args)
    with swept():
        test(idw, *args)
