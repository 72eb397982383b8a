"""The Python binding's own checks (no GPU needed: a call is refused before it
reaches the library), and the forms of the stream argument on a GPU."""
import pytest

from paper_2608_09388_gb300 import hc

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


def test_binding_refuses_arguments():
    f, i = torch.zeros((4, 8)), torch.zeros((4,), dtype=torch.int32)
    m = torch.zeros((2, 10), dtype=torch.uint8)
    with pytest.raises(ValueError):  # [B, V] wanted
        hc.hc_mask_compact(m[0], i, i, i, i)
    with pytest.raises(ValueError):  # pageable host memory
        hc.hc_mask_compact(m, i, i, i, i)
    with pytest.raises(TypeError):  # not a tensor
        hc.hc_mask_compact([[0, 1]], i, i, i, i)
    with pytest.raises(TypeError):  # a required tensor missing
        hc.hc_sparse_linear_fwd(f, i, None, None, 0, f)
    with pytest.raises(TypeError):  # only fp32 and bf16
        hc.hc_sparse_linear_fwd(f.half(), i, f, None, 0, f)
    with pytest.raises(IndexError):  # W [K, C_out] wanted
        hc.hc_sparse_linear_fwd(f, i, f[0], None, 0, f)


@pytest.mark.gpu
def test_binding_streams():
    """The current stream, a stream object and a raw handle order the work."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    side = torch.cuda.Stream()
    alpha = torch.tensor([0.5, 3.0, -1.0, 2.0], device="cuda")
    torch.cuda.synchronize()
    for how in (None, side, side.cuda_stream, 0):
        sel = torch.full((2,), -7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            hc.hc_mask_select_topk(alpha, 2, sel, stream=how)
        torch.cuda.synchronize()
        assert sel.tolist() == [1, 3], how
    with pytest.raises(ValueError):  # not contiguous
        hc.hc_mask_select_topk(alpha[::2], 1, sel)
    with pytest.raises(hc.HcError):
        hc.hc_mask_select_topk(alpha, 9, sel)
