"""Device arrays of cs_set_instances: read by a kernel only where they hold
all n instances, refused otherwise as a copy past an allocation is."""
import ctypes as C

import numpy as np
import pytest

from paper_2501_17792_gb300 import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def alloc():
    torch.zeros(1, device="cuda")
    try:
        rt = C.CDLL("libcudart.so.13")
    except OSError:
        pytest.skip("no CUDA runtime library to allocate with")
    made = []

    def make(data, n_bytes):
        p = C.c_void_p()
        assert rt.cudaMalloc(C.byref(p), C.c_size_t(n_bytes)) == 0
        made.append(p)
        assert rt.cudaMemcpy(p, C.c_void_p(data.ctypes.data), C.c_size_t(min(n_bytes, data.nbytes)), 1) == 0
        return p

    yield make
    torch.cuda.synchronize()
    for p in made:
        rt.cudaFree(p)


@pytest.mark.parametrize("short", [None, 0, 1, 2])
@pytest.mark.parametrize("n", [2, 5])
def test_arrays_of_their_own_allocations(alloc, n, short):
    """Each array in an allocation that holds exactly n instances, or one of
    them one fewer (the rest of its memory block is mapped either way)."""
    from paper_2501_17792_gb300 import binding
    sc = S.crowd(n_templates=1, n_gauss=300, sh_degree=0, cols=n, rows=1, width=64, height=48)
    inst = [np.ascontiguousarray(a) for a in (sc.instances.template_id.astype(np.int32),
                                              sc.instances.root.astype(np.float32), sc.instances.pose.astype(np.float32))]
    r = binding.Renderer(device=0)
    r.upload_templates(sc.templates)
    r.set_lod(sc.lod)
    r.set_instances(*inst)
    want = r.render(sc.camera).clone()
    ptr = [alloc(a, a.nbytes // n * (n - (k == short))) for k, a in enumerate(inst)]
    rc = r.L.cs_set_instances(r.h, n, *ptr, 1)
    assert rc == (binding.CS_OK if short is None else binding.CS_ERR_CUDA)
    # the context goes on
    if short is None:
        assert torch.equal(r.render(sc.camera), want)
    r.set_instances(*[torch.from_numpy(a).cuda() for a in inst])
    assert torch.equal(r.render(sc.camera), want)
    r.close()
