"""The mixed form rounds a tracer once per stage: absolute tracers (meshes with
partial bottom cells hold no anomalies) lose no more of their FP32 precision
in a step than that.

One rounding to FP32 is off by at most 2^-24 of the value, 2^-24 / sqrt(3)
rms.  A step rounds the input, each stage's result, which enters the step's
with its Runge-Kutta weight (SSPRK2: 1/2; SSPRK3: 1/4 x 2/3 and 2/3), and the
result: rms errors of sqrt(1 + 1/4 + 1) and sqrt(1 + 1/36 + 4/9 + 1) of those.
Forming h phi and combining it rounds twice more a stage and exceeds that."""
import numpy as np
import pytest

import oracle
from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


@pytest.mark.parametrize("order,roundings", [(2, 2.25), (3, 1.0 + 1.0 / 36 + 4.0 / 9 + 1.0)])
def test_a_step_rounds_a_tracer_once_per_stage(order, roundings):
    m, L, p, (u, h, tr), layers = inputs.partial_case(
        40, 48, 10e3, 12, depth=lambda x, y: 150.0 + 800.0 * y / y.max(), nTracers=2)
    kw = dict(max_level=layers[0], rest_thickness=layers[1])
    _, _, ref = oracle.Oracle(m, L, p, **kw).step(order, 100.0, 10, u, h, tr, n_steps=1)
    dm = binding.Mesh(m, L, **kw)
    st = binding.State(dm, p, "mixed")
    st.load_state(u, h, tr)
    st.step(order, 100.0, 10, 1)
    _, _, got = st.read_state()
    st.close()
    dm.close()
    wet = np.arange(L)[None, :] < layers[0][:, None]
    for a, b in zip(got, ref):
        rms = np.sqrt(np.mean((a[wet] / b[wet] - 1.0) ** 2))
        assert rms <= 2.0 ** -24 / np.sqrt(3.0) * np.sqrt(roundings), rms
