"""Packed launches take the largest baroclinic patches that fit, whatever the
state's own are, and keep the bits."""
import numpy as np
import pytest

from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("bcl_patch_cells", [0, 96])
def test_packed_patches(precision, bcl_patch_cells):
    # 38,000 cells: the state's own patches are waves of 125 cells, its thickness
    # patches full-sized (and so those of packed launches too)
    m, L, p, state = inputs.channel_case(190, 200, 5e3, 2, perturb=True)
    dm = binding.Mesh(m, L)
    sts = []
    for _ in range(2):
        st = binding.State(dm, p, precision, bcl_patch_cells=bcl_patch_cells)
        st.load_state(*state)
        sts.append(st)
    own = binding.plan_bytes(dm)
    binding.step_batch(sts[:1], 3, [60.0], [6], 2)
    # a second plan for packed launches, unless the state asked for its size
    assert (binding.plan_bytes(dm) > own) == (bcl_patch_cells == 0)
    sts[1].step(3, 60.0, 6, 2)
    for a, b in zip(sts[0].read_state(), sts[1].read_state()):
        assert np.array_equal(a, b)
    for st in sts:
        st.close()
    dm.close()
