"""A row with more edges than there are items (some item must repeat) is refused
before its slice of 32 rows padded to that length is laid out."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_overlong_row_is_refused_without_its_layout(dlm_lib):
    J, d = 1000, 20_000_000  # 6.4 GB padded
    dev = torch.device("cuda")
    rp = torch.tensor([0, d, d + 2], dtype=torch.int64, device=dev)
    col = (torch.arange(d + 2, device=dev) % J).to(torch.int32)
    c = torch.full((d + 2,), -1.0, device=dev)
    b = torch.ones(J, dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    dlm_lib.dlm_release_cached_memory()
    before = torch.cuda.mem_get_info()[0]
    with pytest.raises(dlm_lib.DlmError) as e:
        dlm_lib.Solver(rp, col, c, c, b, J)
    assert e.value.status == dlm_lib.DLM_ERR_INVALID_ARG and "twice" in str(e.value)
    assert before - torch.cuda.mem_get_info()[0] < 1 << 30
