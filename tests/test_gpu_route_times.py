"""Calls that a kernel made for larger or sparser ones must not slow down: each
against a call of the same kind that takes the other kernel or is larger."""
import pytest

from paper_2608_09388_gb300 import hc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


def us(f):
    from _timing import device_us
    return device_us(f)


def count(n):
    return torch.tensor([n], dtype=torch.int32, device="cuda")


def neighbours(L, n):
    g = torch.Generator("cuda").manual_seed(L)
    return torch.stack([torch.randperm(n, generator=g, device="cuda") for _ in range(L)]).int()


def conv_us(L, n, ci, co, dtype=torch.float32):
    x, W = torch.randn((n, ci), device="cuda"), torch.randn((L * ci, co), device="cuda")
    x, W = x.to(dtype), W.to(dtype)
    y, rb, c = torch.empty((n, co), dtype=dtype, device="cuda"), neighbours(L, n), count(n)
    return us(lambda: hc.hc_sparse_conv_rulebook_fwd(x, rb, c, W, None, hc.HC_ACT_ELU, y))


def test_fp32_conv_of_few_channels():
    """32 slots of 3 channels are 1.5 steps of 64, not 3.5 times 9 slots'."""
    t9, t32 = conv_us(9, 41920, 3, 64), conv_us(32, 41920, 3, 64)
    assert t32 < 2 * t9, (t9, t32)


def test_fp32_dense_layer_of_few_channels():
    """4 of 48 channels: not two fifths of the time."""
    def dense(ci):
        x = torch.randn((64, 655, ci), device="cuda")
        W, sp = torch.randn((9 * ci, 64), device="cuda"), neighbours(9, 655).t().contiguous()
        y = torch.empty((64, 655, 64), device="cuda")
        return us(lambda: hc.hc_spiral_conv_fwd(x, sp, W, None, hc.HC_ACT_ELU, y))
    few, many = dense(4), dense(48)
    assert few < 0.31 * many, (few, many)


def head_us(n, ci, co, dtype):
    x, W = torch.randn((n, ci), device="cuda").to(dtype), torch.randn((ci, co), device="cuda").to(dtype)
    y, c = torch.empty((n, co), dtype=dtype, device="cuda"), count(n)
    return us(lambda: hc.hc_sparse_linear_fwd(x, c, W, None, hc.HC_ACT_NONE, y))


def test_small_linear_heads():
    """655 rows: a bf16 head of 60 outputs takes no longer than a one-slot conv of
    as many channels, which takes the 64 x 64 tiles (1.4 times as long on the
    narrow-head kernel); an fp32 head of 16 outputs no longer than one of 3 (1.5
    times)."""
    head, tiles = head_us(655, 64, 60, torch.bfloat16), conv_us(1, 655, 64, 60, torch.bfloat16)
    assert head < 1.2 * tiles, (head, tiles)
    many, few = (head_us(655, 128, co, torch.float32) for co in (16, 3))
    assert many < 1.2 * few, (many, few)


def test_mapping_of_many_small_frames():
    """16 KB of masks in one-vertex frames: a wave of CTAs that each count the whole
    mask takes a fifth longer than the count pass, which one byte more brings."""
    def mapping(B):
        i32 = dict(dtype=torch.int32, device="cuda")
        mask = (torch.arange(B, device="cuda") % 2).to(torch.uint8).view(B, 1)
        spiral = torch.zeros((1, 1), **i32)
        out = [torch.empty(s, **i32) for s in ((B, 2), (B, 1), (B + 1,), (1,), (1, B))]
        return us(lambda: hc.hc_mask_compact_rulebook(mask, spiral, hc.HC_LAYOUT_DENSE, *out))
    below, above = mapping(16384), mapping(16400)
    assert below < 1.12 * above, (below, above)


def test_input_gradient_of_few_or_odd_channels():
    """dx alone, every tap present, against 64 -> 64 channels: 16 input channels in
    bf16 (0.87 of it with a tile of 64 to a slot), 3 in fp32 (0.78), and 42 outputs
    in bf16 (2.4 times on the CUDA cores)."""
    L, n = 9, 41920
    rb, c = neighbours(L, n), count(n)
    ptr = torch.empty((n + 1,), dtype=torch.int32, device="cuda")
    taps = torch.empty((L * n,), dtype=torch.int32, device="cuda")
    hc.hc_conv_rulebook_transpose(rb, c, n, ptr, taps)

    def dx_us(ci, co, dtype):
        x, W = (torch.randn(s, device="cuda").to(dtype) for s in ((n, ci), (L * ci, co)))
        y, dy = (torch.randn((n, co), device="cuda").to(dtype) for _ in "ab")
        return us(lambda: hc.hc_sparse_conv_rulebook_bwd(x, rb, c, W, y, dy, hc.HC_ACT_ELU, ptr,
                                                         taps, torch.empty_like(x)))
    for dtype, ci, co, most in ((torch.bfloat16, 16, 64, 0.75), (torch.bfloat16, 64, 42, 1.6),
                                (torch.float32, 3, 64, 0.5)):
        t, base = dx_us(ci, co, dtype), dx_us(64, 64, dtype)
        assert t < most * base, (dtype, ci, co, t, base)


def test_weight_gradient_of_few_channels():
    """3 of 64 input channels in fp32 are not as much work as 64 (0.99 of their time
    with one tile width)."""
    L, n = 9, 41920
    rb, c = neighbours(L, n), count(n)

    def dW_us(ci):
        x, y, dy = (torch.randn(s, device="cuda") for s in ((n, ci), (n, 64), (n, 64)))
        dW = torch.empty((L * ci, 64), device="cuda")
        return us(lambda: hc.hc_sparse_conv_rulebook_bwd(x, rb, c, dW, y, dy, hc.HC_ACT_ELU, None,
                                                         None, None, dW, None))
    few, many = dW_us(3), dW_us(64)
    assert few < 0.75 * many, (few, many)
