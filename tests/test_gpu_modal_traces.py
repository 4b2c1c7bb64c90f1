"""The memory of the modal traces: taken for a call and given back after it, so that whatever fitted beside a context
without them still fits; declined, refused or absent, the states stay the same bit for bit."""
import numpy as np
import pytest

from oracle import to_abi
from synthetic import periodic_cube_mesh, rock_material
from synthetic.mesh import FACE_BC_ABSORBING, FACE_BC_FREE_SURFACE

from parity_util import make_solver
from test_gpu_boundary import _box, _rough_state
from test_gpu_picard import _material

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import paper_2502_09714_gb300 as dgpkg
    dgpkg.build()
    dgpkg.load_library()


class _Counting:
    """Allocator that knows what is held, and refuses the next `refuse` requests."""

    def __init__(self):
        import paper_2502_09714_gb300 as dgpkg
        self.base = dgpkg.torch_allocator()
        self.live, self.asked, self.refuse = {}, [], 0
        self.allocator = dgpkg.torch_allocator()
        self.allocator.alloc = type(self.base.alloc)(self._alloc)
        self.allocator.free = type(self.base.free)(self._free)

    def _alloc(self, nbytes, stream, user):
        self.asked.append(nbytes)
        if self.refuse > 0:
            self.refuse -= 1
            return None
        p = self.base._keep[0](nbytes, stream, user)
        if p:
            self.live[p] = nbytes
        return p

    def _free(self, ptr, nbytes, stream, user):
        del self.live[ptr]
        self.base._keep[1](ptr, nbytes, stream, user)

    @property
    def held(self):
        return sum(self.live.values())


def _problem(N, n=3, seed=5):
    mesh = periodic_cube_mesh(n, 4000.0, jitter=0.1, seed=seed)
    return mesh, rock_material(mesh.n_elem, cd=2e-6), to_abi(_rough_state(mesh.n_elem, N, seed=seed))


def _solver(mesh, mat, N, allocator=None):
    import paper_2502_09714_gb300 as dgpkg
    s = dgpkg.Solver(mesh.elem_xyz, mesh.elem_vid, N, allocator=allocator)
    s.set_material(mat)
    return s


def _step(s, Q):
    s.set_state(Q)
    s.step(2, 0.5 * s.dt)
    return s.get_state()[0]


@pytest.mark.parametrize("N", [1, 2, 3, 4])
def test_held_during_the_call_only(N):
    mesh, mat, Q = _problem(N)
    c = _Counting()
    s = _solver(mesh, mat, N, c.allocator)
    s.set_state(Q)
    before, c.asked = c.held, []
    s.step(1, 0.25 * s.dt)
    assert s.modal_trace_bytes > 0 and c.asked == [s.modal_trace_bytes]
    assert c.held == before
    s.set_receivers(mesh.elem_xyz[:2].mean(axis=1))
    s.step(1, 0.25 * s.dt)
    before = c.held
    s.adjoint_gradient(np.zeros((2, 2, 3)), 2, 0.25 * s.dt, snapshots=2)
    assert s.modal_trace_bytes > 0 and c.held == before
    q = np.ascontiguousarray(Q, dtype=np.float32)
    s.step_host(q, np.empty_like(q), 0.25 * s.dt)
    before = c.held
    s.step_host(q, np.empty_like(q), 0.25 * s.dt)
    assert s.modal_trace_bytes > 0 and c.held == before
    s.close()
    assert c.held == 0


def test_the_picard_predictor_and_the_step_without_allocation_do_not_ask():
    import torch
    mesh, mat, Q = _problem(2)
    c = _Counting()
    s = _solver(mesh, mat, 2, c.allocator)
    s.set_predictor("picard", 1)
    s.set_state(Q)
    c.asked = []
    s.step(1, 0.25 * s.dt)
    assert s.modal_trace_bytes == 0 and c.asked == []
    s.set_predictor("ck")
    qa = torch.from_numpy(np.ascontiguousarray(Q, dtype=np.float32)).cuda()
    s.step_noalloc(qa, torch.empty_like(qa), 0.25 * s.dt)
    torch.cuda.synchronize()
    assert c.asked == []
    s.close()


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("allocator", [False, True])
def test_declined_and_refused(N, allocator):
    """No limit, a limit below the traces' size, none at all, and a refusal, which counts for its call only."""
    mesh, mat, Q = _problem(N)
    c = _Counting()
    s = _solver(mesh, mat, N, c.allocator if allocator else None)
    q = _step(s, Q)
    full = s.modal_trace_bytes
    assert full > 0
    for limit in (0, full - 1, full, -1):
        s.set_modal_traces(limit)
        np.testing.assert_array_equal(_step(s, Q), q)
        assert s.modal_trace_bytes == (full if limit in (full, -1) else 0)
    if allocator:
        s.set_state(Q)
        c.refuse = 1
        s.step(1, 0.5 * s.dt)
        assert c.refuse == 0 and s.modal_trace_bytes == 0
        s.step(1, 0.5 * s.dt)
        assert s.modal_trace_bytes == full
        np.testing.assert_array_equal(s.get_state()[0], q)
    s.close()


def test_other_allocations_get_the_kept_memory():
    """After a step, a tensor of more than the memory that is free, by half of the traces' size, still fits."""
    import torch
    mesh, mat, Q = _problem(4, n=16)                    # 24,576 tets, traces of 113 MB
    torch.cuda.empty_cache()
    s = _solver(mesh, mat, 4)
    _step(s, Q)
    s.step(1, 0.5 * s.dt)
    assert s.modal_trace_bytes > 100e6
    free, _ = torch.cuda.mem_get_info()
    x = torch.empty(free + s.modal_trace_bytes // 2, dtype=torch.uint8, device="cuda")
    assert x.numel() > free
    del x
    torch.cuda.empty_cache()
    s.step(1, 0.5 * s.dt)                               # and the traces are there again
    assert s.modal_trace_bytes > 100e6
    s.close()


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_both_paths_with_boundaries_over_several_rounds(N):
    """5,400 tets with outer faces, above the size from which degree 5 takes the traces (one face staged at a time):
    the whole state with and without them."""
    import torch
    mesh = _box((10, 10, 9), (False, False, False), FACE_BC_FREE_SURFACE, FACE_BC_ABSORBING, seed=N)
    least = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    assert mesh.n_elem >= least
    mat = _material("cdm", mesh.n_elem, np.random.default_rng(N))
    Q = to_abi(_rough_state(mesh.n_elem, N, seed=N))
    s = make_solver(mesh, mat, N)
    q = _step(s, Q)
    assert s.modal_trace_bytes > 0
    s.set_modal_traces(0)
    np.testing.assert_array_equal(_step(s, Q), q)
    assert s.modal_trace_bytes == 0
    assert np.isfinite(q).all() and np.abs(q - Q).max() > 0
    s.close()


def test_small_meshes_of_degree_5_run_without():
    mesh, mat, Q = _problem(5)
    s = _solver(mesh, mat, 5)
    _step(s, Q)
    assert s.modal_trace_bytes == 0
    s.set_modal_traces(1 << 40)
    _step(s, Q)
    assert s.modal_trace_bytes == 0
    s.close()
