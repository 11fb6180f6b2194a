"""The device memory that component calls keep between them is given back on request, and (by the driver) to a plan
that does not fit beside it."""
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

    desc = q.make_desc(4, 128, "fp32", 48, outputs=["GR_diag"])
    assert 300 * MB < q.footprint(desc) < 400 * MB, q.footprint(desc) / MB
    q.zgemm_batched(A, A, "emu64")
    filler = torch.empty(free() - 180 * MB, dtype=torch.uint8, device="cuda")
    try:
        plan = q.Plan(desc)
        plan.close()
    finally:
        del filler
        torch.cuda.empty_cache()
