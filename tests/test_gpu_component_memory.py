"""The device memory that component calls keep between them, and its return on request."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2606_25595_gb300 import build
    build.build()
    import paper_2606_25595_gb300 as q
    q.load()
    return q


def test_kept_memory_is_given_back(q):
    import torch
    MB = 1 << 20
    A = torch.randn(64, 256, 256, dtype=torch.complex128, device="cuda")
    free = lambda: (torch.cuda.synchronize(), torch.cuda.empty_cache(), torch.cuda.mem_get_info()[0])[2]  # noqa: E731
    C = q.zgemm_batched(A, A, "emu64")  # 300 MB of digit planes
    assert torch.equal(C, C.clone())  # (kernels are loaded at their first use)
    q.release_memory()
    base = free()
    assert torch.equal(q.zgemm_batched(A, A, "emu64"), C)
    assert base - free() >= 200 * MB
    q.release_memory()
    assert base - free() <= 64 * MB
    q.release_memory()  # an empty pool


def test_contact_on_its_own_takes_the_decimation_s_blocks_only(q):
    """Twelve blocks per energy (ten of the iteration, the inverse's two), and no digit planes or refinement areas."""
    import torch
    n, ne = 40, 400
    H00 = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    H01 = torch.eye(n, dtype=torch.complex128, device="cuda") * 0.5
    E = torch.linspace(-0.5, 0.5, ne, dtype=torch.float64, device="cuda")
    free = lambda: (torch.cuda.synchronize(), torch.cuda.empty_cache(), torch.cuda.mem_get_info()[0])[2]  # noqa: E731
    S, st = q.lead_self_energy(H00, H01, E, 1e-3)
    assert not st.any()
    q.release_memory()
    base = free()
    S2, st = q.lead_self_energy(H00, H01, E, 1e-3)
    assert torch.equal(S, S2)
    assert base - free() <= 12 * ne * n * n * 16 + (64 << 20)
