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


def test_fp64_without_tensor_memory_takes_the_global_subcycle(monkeypatch):
    """SSE_BTR_TMEM=0 on the 92,480-cell channel, whose FP64 patches fit an SM
    only with their edge data in tensor memory: the global-memory sub-cycle
    runs, within the FP64 parity bound of the oracle."""
    import oracle
    m, L, p, (u, h, tr), run = inputs.workload("channel_1km", perturb=True, L=2)
    o = oracle.Oracle(m, L, p)
    ubar, _ = o.split(u, h)
    G = 1e-6 * np.sin(np.arange(m.nEdges) * 0.37)
    u1, Fz, _ = o.barotropic_substep(3, ubar, o.ssh(h), G, run["dt"], 8)
    monkeypatch.setenv("SSE_BTR_TMEM", "0")
    dm = binding.Mesh(m, L)
    st = binding.State(dm, p, "fp64")
    assert st.subcycle_shape() == (0, False) and st.patches() == 0
    st.load_state(u, h, tr)
    st.set("ubar", ubar)
    st.set("G", G)
    st.barotropic_substep(3, run["dt"], 8)
    for f, ref in (("ubar", u1), ("Fzeta", Fz)):
        assert np.linalg.norm(st.get(f) - ref) < 1e-11 * np.linalg.norm(ref)
    st.close()
    dm.close()
