"""gs_copy_arrays: several device arrays copied in one launch, byte for byte."""
import pytest
import torch

from paper_2507_15683_gb300 import gsr

pytestmark = pytest.mark.gpu


def copy(items):
    gsr.gs_copy_arrays([d.data_ptr() for d, _ in items], [s.data_ptr() for _, s in items],
                       [s.numel() for _, s in items], torch.cuda.current_stream().cuda_stream)


# sizes around the 16-byte step and the loop with four loads in flight, at
# addresses that allow 16 bytes on both ends, on one, and on none
@pytest.mark.parametrize("off_d,off_s", [(0, 0), (16, 32), (0, 4), (1, 0), (8, 8)])
def test_bytes_arrive_and_nothing_else_changes(off_d, off_s):
    sizes = [0, 1, 15, 16, 17, 4095, 4096, 4097, 12_000_005]
    g = torch.Generator(device="cuda").manual_seed(5)
    src = [torch.randint(0, 256, (n + off_s,), dtype=torch.uint8, device="cuda", generator=g)[off_s:] for n in sizes]
    full = [torch.full((off_d + n + 32,), 7, dtype=torch.uint8, device="cuda") for n in sizes]
    copy([(f[off_d:off_d + n], s) for f, s, n in zip(full, src, sizes)])
    for f, s, n in zip(full, src, sizes):
        assert torch.equal(f[off_d:off_d + n], s)
        assert bool((f[:off_d] == 7).all()) and bool((f[off_d + n:] == 7).all())


def test_bad_arguments_are_errors():
    s = torch.zeros(4, dtype=torch.uint8, device="cuda")
    gsr.gs_copy_arrays([], [], [], 0)
    gsr.gs_copy_arrays([0], [0], [0], 0)
    for dst, src, n in [([0], [s.data_ptr()], [4]), ([s.data_ptr()], [0], [4]), ([s.data_ptr()], [s.data_ptr()], [-1]),
                        ([s.data_ptr()] * 17, [s.data_ptr()] * 17, [0] * 17)]:
        with pytest.raises(gsr.GsError):
            gsr.gs_copy_arrays(dst, src, n, 0)
