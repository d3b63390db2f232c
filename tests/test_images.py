"""Accumulation of several feature images in one pass: the bits of one
accumulation per image, and its argument checks (no GPU)."""
import pytest
import torch

from paper_2403_16862_gb300 import api, build


@pytest.fixture(scope="module")
def B():
    build.build()
    from paper_2403_16862_gb300 import _binding
    _binding.load()
    yield _binding
    _binding.inpc_set_fault(None)


def test_arguments_are_checked(B):
    fake = 1 << 20  # never dereferenced
    for images, n, acc, dtype in [([], 8, fake, B.INPC_F32), ([fake] * 5, 8, fake, B.INPC_F32),
                                  ([fake, None], 8, fake, B.INPC_F32), ([fake], 8, None, B.INPC_F32),
                                  ([fake], -1, fake, B.INPC_F32), ([fake + 1], 8, fake, B.INPC_BF16),
                                  ([fake], 8, fake + 2, B.INPC_F32)]:
        with pytest.raises(B.InpcError) as e:
            B.inpc_accumulate_images(images, dtype, n, 0.5, True, acc, None)
        assert e.value.status == B.INPC_ERR_INVALID_ARG
    with pytest.raises(B.InpcError) as e:
        B.inpc_accumulate_images([fake], 7, 8, 0.5, True, fake, None)
    assert e.value.status == B.INPC_ERR_UNSUPPORTED
    B.inpc_set_fault("corrupt_args")
    try:
        with pytest.raises(B.InpcError) as e:
            B.inpc_accumulate_images([fake], B.INPC_F32, 8, 0.5, True, fake, None)
        assert e.value.status == B.INPC_ERR_INVALID_ARG
    finally:
        B.inpc_set_fault(None)


@pytest.mark.gpu
@pytest.mark.parametrize("n,k,offset", [(1, 1, 0), (3, 2, 0), (4, 3, 0), (4_099, 4, 0), (70_001, 4, 1),
                                        (20_000_003, 2, 0)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_same_bits_as_one_by_one(gpu, B, n, k, offset, dtype):
    images = [torch.randn(n + offset, device=gpu).to(dtype)[offset:] for _ in range(k)]
    for fresh in (True, False):
        want = torch.randn(n + offset, device=gpu)[offset:].contiguous() if not fresh else torch.zeros(n, device=gpu)
        got = torch.full((n,), float("nan"), device=gpu) if fresh else want.clone()
        for im in images:
            B.inpc_accumulate_image(im.data_ptr(), B.INPC_F32 if dtype == torch.float32 else B.INPC_BF16, n, 1.0 / 3,
                                    want.data_ptr(), api._stream())
        B.inpc_accumulate_images([im.data_ptr() for im in images],
                                 B.INPC_F32 if dtype == torch.float32 else B.INPC_BF16, n, 1.0 / 3, fresh,
                                 got.data_ptr(), api._stream())
        assert torch.equal(got, want)
