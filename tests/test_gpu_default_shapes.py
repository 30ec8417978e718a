"""The default launch shapes follow one rule over all sizes and precisions:
the sub-cycle takes one patch per 64 cells (one per SM at most), so that
neither the precision nor one more row of cells changes how a small mesh is
cut."""
import pytest

from paper_2105_13484_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.load()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (8, 18), (12, 20), (16, 30), (16, 32), (19, 28),
                                   (24, 44)])
def test_small_meshes_take_one_patch_per_64_cells(nx, ny, precision):
    m, L, p, _ = inputs.channel_case(nx, ny, 10e3, 3)
    dm = binding.Mesh(m, L)
    st = binding.State(dm, p, precision)
    assert st.patches() == m.nCells // 64
    st.close()
    dm.close()
