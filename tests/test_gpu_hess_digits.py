"""The digits of the FP32 Hessian evaluation, against the FP64 one, on draws of the measured
workloads (a field of 500 sources, a crowded region of 64), as geometric means over the draws:
  * the median source's gradient error on the field: 1.95e-7 with the star's terms in the
    pixel frame, 2.29e-7 with them in FP32 whitened coordinates;
  * the error of the Hessian's 2 x 2 block of a source's type probabilities in the crowd: 1.4e-7
    with d/da_i summed as one term, 2.9e-7 with its two parts scaled apart in FP64.
Each bound is the geometric middle of the two."""
import math

import pytest

pytestmark = pytest.mark.gpu


def _pairs(name, fp32_case, seeds):
    import torch
    from paper_1801_10277_gb300 import celeste as cel
    from perf import cases
    for seed in seeds:
        s = cases.prepare(fp32_case, seed)
        f32 = cases.run(s)[name].double().reshape(fp32_case["n_src"], -1)
        s["precision"] = cel.FP64
        f64 = cases.run(s)[name].reshape(fp32_case["n_src"], -1).clone()
        torch.cuda.synchronize()
        s["problem"].close()
        yield f32, f64


def _mean(values):
    return math.exp(sum(map(math.log, values)) / len(values))


def test_gradient_digits_of_a_field():
    case = dict(layout="field", call="hess", fp32=True, width=2048, height=1489, n_src=500, bright=0.0)
    errors = [float(((g - e).norm(dim=1) / e.norm(dim=1)).median()) for g, e in _pairs("grad", case, range(11, 15))]
    assert _mean(errors) <= 2.11e-7, errors


def test_type_probability_digits_in_a_crowd():
    case = dict(layout="crowded", call="hess", fp32=True, side=256, n_src=64)
    errors = []
    for h, e in _pairs("hess", case, range(21, 31)):
        h, e = (x.view(-1, 44, 44)[:, 26:28, 26:28] for x in (h, e))
        errors.append(float((h - e).norm() / e.norm()))
    assert _mean(errors) <= 2.05e-7, errors
