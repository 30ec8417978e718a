"""Device memory of the patch plans: one copy shared by a mesh's states, found
again by the states that follow, and nothing left of sse_tune's candidates."""
import numpy as np
import pytest

from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


def test_states_share_the_plans():
    m, L, p, state = inputs.channel_case(16, 32, 10e3, 4, perturb=True)
    dm = binding.Mesh(m, L)
    assert binding.plan_bytes(dm) == 0
    a = binding.State(dm, p, "mixed")
    one = binding.plan_bytes(dm)
    assert one > 0
    b = binding.State(dm, p, "mixed")
    assert binding.plan_bytes(dm) == one
    c = binding.State(dm, p, "fp64")
    both = binding.plan_bytes(dm)
    assert both > one
    # the states that stay keep working when the one that made the plans goes
    for st in (a, b):
        st.load_state(*state)
        st.step(3, 100.0, 6, 2)
    ref = a.read_state()
    a.close()
    assert binding.plan_bytes(dm) == both
    d = binding.State(dm, p, "mixed")
    d.load_state(*state)
    d.step(3, 100.0, 6, 2)
    for st in (b, d):
        for x, y in zip(st.read_state(), ref):
            assert np.array_equal(x, y)
    for st in (b, c, d):
        st.close()
    for _ in range(3):
        with_one = binding.State(dm, p, "mixed")
        assert binding.plan_bytes(dm) == both
        with_one.close()
    dm.close()


def test_a_state_may_outlive_its_mesh_handle():
    m, L, p, _ = inputs.channel_case(16, 32, 10e3, 4)
    dm = binding.Mesh(m, L)
    st = binding.State(dm, p, "mixed")
    dm.close()
    st.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_tuning_leaves_no_plans_behind(precision):
    m, L, p, _ = inputs.channel_case(48, 60, 10e3, 4)
    dm = binding.Mesh(m, L)
    st = binding.State(dm, p, precision)
    before = binding.plan_bytes(dm)
    binding.tune_shapes(dm, p, precision, "throughput")
    assert binding.plan_bytes(dm) == before
    st.close()
    dm.close()
    dm = binding.Mesh(m, L)
    binding.tune_shapes(dm, p, precision, "latency")
    assert binding.plan_bytes(dm) == 0
    dm.close()
