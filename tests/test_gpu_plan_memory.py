"""Device memory of the patch plans: one copy shared by a mesh's states, found
again by the states that follow, and nothing left of sse_tune's rejected
candidates."""
import ctypes as ct

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
def test_tuning_leaves_the_chosen_plans_only(precision):
    m, L, p, state = inputs.channel_case(48, 60, 10e3, 4, perturb=True)
    dm = binding.Mesh(m, L)
    for objective in ("throughput", "latency"):
        before = binding.plan_bytes(dm)
        shapes = binding.tune_shapes(dm, p, precision, objective)
        after = binding.plan_bytes(dm)
        # a state of these shapes, alone and packed, finds all it needs ...
        st = binding.State(dm, p, precision, **shapes)
        st.load_state(*state)
        binding.step_batch([st], 3, [100.0], [6], 1)
        assert binding.plan_bytes(dm) == after
        st.close()
        # ... and nothing else was left
        fresh = binding.Mesh(m, L)
        st = binding.State(fresh, p, precision, **shapes)
        st.load_state(*state)
        binding.step_batch([st], 3, [100.0], [6], 1)
        assert after - before <= binding.plan_bytes(fresh)
        st.close()
        fresh.close()
    dm.close()


def _used():
    """Bytes in use in the device's memory pool, from which states and plans come."""
    rt = ct.CDLL("libcudart.so.13")
    pool, out = ct.c_void_p(), ct.c_uint64()
    assert rt.cudaDeviceSynchronize() == 0
    assert rt.cudaDeviceGetDefaultMemPool(ct.byref(pool), 0) == 0
    assert rt.cudaMemPoolGetAttribute(pool, 7, ct.byref(out)) == 0   # cudaMemPoolAttrUsedMemCurrent
    return out.value


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("nx,ny", [(16, 32), (48, 60)])
def test_footprint_covers_the_state_and_its_plans(nx, ny, precision):
    m, L, p, state = inputs.channel_case(nx, ny, 10e3, 4, perturb=True)
    dm = binding.Mesh(m, L)
    fp = binding.footprint(dm, p, precision)
    assert binding.plan_bytes(dm) == 0
    before = _used()
    a = binding.State(dm, p, precision)
    a.load_state(*state)
    binding.step_batch([a], 3, [100.0], [6], 1)
    took = _used() - before
    # the pool rounds each of about 120 arrays up to 512 bytes, the count to 256
    assert fp - 120 * 512 <= took <= fp + 120 * 512, (took, fp)
    a.close()
    dm.close()


def test_idle_plans_stay_inside_a_servers_budget():
    cases = []
    for nx, ny in ((48, 60), (40, 66)):
        m, L, p, state = inputs.channel_case(nx, ny, 10e3, 4, perturb=True)
        cases.append((binding.Mesh(m, L), p, state))

    def run(budget):
        srv = binding.Server(hbm_budget=budget, max_active=2)
        for dm, p, (u, h, tr) in cases:
            r = srv.submit(dm, p, "mixed", u, h, tr, 3, 100.0, 6, 2)
            assert r.wait(120)["status"] == "done"
        srv.close()
        return [binding.plan_bytes(dm) for dm, _, _ in cases]

    ample = run(1 << 30)
    assert ample[0] > 0 and ample[1] > 0                # found again by the next request
    budget = max(binding.footprint(dm, p, "mixed") for dm, p, _ in cases) + min(ample) // 2
    left = run(budget)
    # the first mesh's idle plans gave way to the second request
    assert left[0] == 0 and left[1] > 0
    for dm, _, _ in cases:
        dm.close()


def test_threads_share_plans_while_others_tune_and_go():
    """States come, step and go on several threads and streams while sse_tune
    frees idle plans of the same mesh: the bits are those of a state alone."""
    import threading

    torch = pytest.importorskip("torch")
    m, L, p, state = inputs.channel_case(48, 60, 10e3, 4, perturb=True)
    dm = binding.Mesh(m, L)
    ref = {}
    for precision in ("mixed", "fp64"):
        st = binding.State(dm, p, precision)
        st.load_state(*state)
        st.step(3, 100.0, 6, 3)
        ref[precision] = st.read_state()
        st.close()
    wrong = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            for i in range(6):
                precision = ("mixed", "fp64")[(i + k) % 2]
                st = binding.State(dm, p, precision, stream=stream.cuda_stream,
                                   patch_cells=(0, 128)[i % 2])
                st.load_state(*state)
                st.step(3, 100.0, 6, 3)
                got = st.read_state()
                st.step(3, 100.0, 6, 3)   # goes with work in flight
                st.close()
                if not all(np.array_equal(a, b) for a, b in zip(got, ref[precision])):
                    wrong.append((k, i))
        except Exception as e:   # noqa: BLE001 - reported by the assertion below
            wrong.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for precision in ("mixed", "fp64"):
        for objective in ("latency", "throughput"):
            binding.tune_shapes(dm, p, precision, objective)
    for t in threads:
        t.join()
    assert not wrong, wrong
    dm.close()
