"""The refinement's error against 64 bits stays where complex volumes had it.

Inputs and 64-bit results are those of perf/cases.py.  The bounds are 1.2 times
the error that passes over whole complex volumes had on these inputs; the half
spectrum with the transforms' constants as plain floats is above each of them
(6.1e-7, 4.0e-7, 3.2e-7)."""
import importlib.util
import os

import pytest

from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def cases(cp):  # noqa: F811
    spec = importlib.util.spec_from_file_location("perf_cases", os.path.join(ROOT, "perf", "cases.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("N,Np,iters,complex_volumes", [
    (128, 80, 50, 3.71e-7),
    (64, 45, 50, 3.05e-7),
    (160, 60, 10, 1.97e-7),
])
def test_error_against_64_bits(cases, N, Np, iters, complex_volumes):
    case = dict(kind="refine", N=N, Np=Np, iters=iters)
    got = cases.run(cases.prepare(case, 3)).real.double()
    ref = cases.exact(case, 3).real
    assert float((got - ref).norm() / ref.norm()) < 1.2 * complex_volumes
