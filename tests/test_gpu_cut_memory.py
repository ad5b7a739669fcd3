"""A reconstruction whose tensor-core operands do not fit in the device's memory
runs without them."""
import numpy as np
import pytest

from test_gpu_cut_steps import sv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_reconstruct_without_room_for_the_digit_planes(sv):  # noqa: F811
    import torch
    # 2^21 x 2^5 outputs: the terms and marginals take some 270 MB, the operands some 540 more
    wa, wb, room = 22, 5, 400 << 20
    gen = torch.Generator(device="cuda").manual_seed(3)
    up = [torch.empty(1 << wa, dtype=torch.float64, device="cuda").exponential_(generator=gen).div_(1 << wa) for _ in range(3)]
    down = [torch.empty(1 << wb, dtype=torch.float64, device="cuda").exponential_(generator=gen).div_(1 << wb) for _ in range(4)]

    def run(out):
        sv.cut_reconstruct(up, down, wa, [wa - 1], wb, keep_mask_a=(1 << (wa - 1)) - 1, keep_mask_b=(1 << wb) - 1, out=out)
        return out

    want, got = (torch.empty(1 << (wa - 1 + wb), dtype=torch.float64, device="cuda") for _ in range(2))
    run(want)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(max(0, free - room), dtype=torch.uint8, device="cuda")
    free, _ = torch.cuda.mem_get_info()
    assert free < 600 << 20
    run(got)
    del filler
    torch.cuda.empty_cache()
    # either form is within 2^-44 of the products: at most four of these sizes
    big = 2 * max(float(u.max()) for u in up) * 4 * max(float(d.max()) for d in down)
    assert float((got - want).abs().max()) <= 2 * 2.0 ** -44 * 4 * big / 2
    assert np.isfinite(float(got.sum()))
