"""sse_tune times the default shapes beside the listed sizes: the shapes it
returns for LATENCY are no slower than what a state that asks for nothing
gets.  The mesh (39,520 cells) is one whose default baroclinic patches, 130
cells, fill one wave of the GPU: 128-cell patches make two, and each listed
size is 25% or more slower."""
import numpy as np
import pytest

from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


def _times(st):
    """Medians over seven steps of the sub-cycle's and the baroclinic stage's time."""
    out = []
    for _ in range(7):
        st.profile(True)
        st.step(3, 60.0, 20, 1)
        r = st.profile_read()
        st.profile(False)
        out.append((r["btr"][0], r["bcl_edge"][0]))
    return np.median(np.array(out[1:]), axis=0)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_tuned_latency_is_no_slower_than_the_default(precision):
    m, L, p, state = inputs.channel_case(190, 208, 5e3, 10, perturb=True)
    dm = binding.Mesh(m, L)
    got = []
    for kw in ({}, binding.tune_shapes(dm, p, precision, "latency")):
        st = binding.State(dm, p, precision, **kw)
        st.load_state(*state)
        got.append(_times(st))
        st.close()
    dm.close()
    # runs of one shape differ by up to 2%
    assert (got[1] <= 1.1 * got[0]).all(), got
