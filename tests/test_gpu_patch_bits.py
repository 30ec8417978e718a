"""sse_tuning.patch_cells keeps the bits: every patch of the tiled sub-cycle
evaluates an edge or a cell with the same arithmetic in the same order,
whichever patch owns it and in whichever launch shape the patch runs (512 or
1024 threads, with or without tensor memory)."""
import numpy as np
import pytest

from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("name,kw,sizes", [("channel_10km", {}, (0, 128, 256, 512)),
                                           ("sphere_l4", {}, (0, 256, 512, 2000)),
                                           ("channel_1km", {"L": 2}, (0, 700, 900))])
def test_subcycle_patch_size_keeps_the_bits(name, kw, sizes, order, precision):
    m, L, p, (u, h, tr), run = inputs.workload(name, perturb=True, **kw)
    dm = binding.Mesh(m, L)
    outs, shapes = [], set()
    for pc in sizes:
        st = binding.State(dm, p, precision, patch_cells=pc)
        assert st.patches() > 0
        shapes.add((st.patches(), st.subcycle_shape()))
        st.load_state(u, h, tr)
        st.step(order, run["dt"] / 2, 8, 2)
        outs.append(st.read_state())
        st.close()
    dm.close()
    assert len(shapes) == len(sizes)
    for o in outs[1:]:
        for a, b in zip(o, outs[0]):
            assert np.array_equal(a, b)
