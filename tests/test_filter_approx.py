"""The FP32 filters with the device's approximate square root and reciprocal in the worst cases of their
specified error: the assertions of the filter tests on a host build that is off by as much.
"""
import os

import pytest

import test_filters as F
from test_filter_units import CSRC, build

APPROX = {"low": "return -1;", "high": "return 1;",
          "mixed": "uint32_t h; memcpy(&h, &x, 4); h *= 2654435761u; return (h >> 30) * (2.0f / 3) - 1;"}


@pytest.fixture(scope="module", params=sorted(APPROX))
def approx(request, tmp_path_factory):
    """The filters with a square root and a reciprocal that are off by 2 u = 2^-23, the device's
    specified error, downwards, upwards or by up to that from value to value."""
    text = open(os.path.join(CSRC, "pm_filter.cuh")).read()
    helper = ("#include <stdint.h>\n#include <string.h>\nstatic inline float off(float x) { %s }\n"
              "static inline float err(float r, float x) {"
              " return (float)((double)r * (1.0 + 0x1p-23 * (double)off(x))); }\n" % APPROX[request.param])
    for old, new in (("return sqrtf(x);", "return err(sqrtf(x), x);"),
                     ("return 1.0f / x;", "return err(1.0f / x, x);"),
                     ("#include <math.h>\n", "#include <math.h>\n" + helper)):
        assert text.count(old) == 1, old
        text = text.replace(old, new)
    return build(tmp_path_factory.mktemp("approx"), text)


@pytest.mark.parametrize("case", F.CASES)
@pytest.mark.parametrize("check", [F.test_filters_decide_only_what_is_certain,
                                   F.test_interpolated_metric_and_its_quality_bound,
                                   F.test_lower_quality_bound], ids=["decide", "metric", "lower"])
def test_bounds_hold_with_approximate_functions(approx, check, case):
    check(approx, *case)
