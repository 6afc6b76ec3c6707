"""The time-out cases that can be started are exactly those that the GPU test runs: a case that once ended in a CUDA
error cannot be launched by hand on a shared GPU either."""
import importlib.util
import os

import pytest

import test_gpu_timeout

HERE = os.path.dirname(os.path.abspath(__file__))


def _case_module():
    spec = importlib.util.spec_from_file_location("timeout_case", os.path.join(HERE, "timeout_case.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_only_the_tested_families_can_be_started():
    case = _case_module()
    marks = test_gpu_timeout.test_expired_wait_reports_timeout_and_leaves_the_context_usable.pytestmark
    tested = next(m.args[1] for m in marks if m.name == "parametrize")
    assert sorted(case.FAMILIES) + ["pack_staged"] == sorted(set(tested) - {"pack_staged"}) + ["pack_staged"]
    with pytest.raises(KeyError):  # before any launch
        case.main("wide")
