"""The bench's account of the gradient (host logic only): a run's result names the form that the library
runs, and the operation count, the launches and the line follow it whatever the launch shapes."""
import argparse

import pytest

import bench
from paper_1712_09434_gb300 import tune
from tests.test_bench_line_cpu import fake_result


def _result(best=None):
    res = dict(fake_result(), adjoint_form=bench.ADJOINT_FORM)
    del res["ms_grad_event_stored"], res["ms_grad_copies_stored"]      # a run times its one form once
    if best:
        res["tuning"] = {"key": "k", "source": "cache", "best": best}
    return res


@pytest.mark.parametrize("best", [None, {"refit_grad": [0, 0, 0]}, {"refit_grad": [64, 8, 0]},
                                  {"refit_grad": [64, 8, 1]}, {"links": [128, 10, 0]}])
def test_stored_states_are_counted_whatever_the_shapes(best):
    line = bench.finish_native(argparse.Namespace(steps=40, warmup=3, events=64), _result(best), 1)
    assert line["adjoint_form_in_step"] == "stored states"
    assert line["stage_tflops"]["refit_grad"] == pytest.approx(
        (bench.FLOP_FWD + bench.FLOP_ADJ) * 25e6 / 2.2e-3 / 1e12)
    assert line["gpu_launches"] == (bench.LAUNCHES_TRACKING + bench.LAUNCHES_REFIT_GRAD["stored states"]) * 40
    assert "stored_states" not in line["adjoint"] and "stored_states" not in line["adjoint"]["batched"]


def test_the_tuner_tries_no_chunk_for_the_gradient():
    assert tune.CANDIDATES["refit_grad"]["chunk"] == [0]
