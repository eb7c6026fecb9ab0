"""An uploaded FP64 operator beyond the persistent kernel's sizes holds its
slices and nothing that no kernel reads: 4 bytes per row pointer, 12 per entry
and 12 per slice (and 8 MB for the allocator's granularity)."""
import pytest
import torch

from workloads import convdiff_2d

pytestmark = pytest.mark.gpu


def test_no_copy_that_nothing_reads(skf):
    A = convdiff_2d(2000, (60.0, 50.0))
    csr = [torch.as_tensor(v, device="cuda") for v in (A.rowptr, A.colind, A.values)]
    first = skf.upload_csr(*csr)   # (one-time allocations)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    op = skf.upload_csr(*csr)
    torch.cuda.synchronize()
    held = free - torch.cuda.mem_get_info()[0]
    slots = 32 * ((A.n + 31) // 32)
    assert held <= 4 * (A.n + 1) + 5 * slots * 12 + 12 * slots // 32 + (8 << 20)
    assert op.csr.n == first.csr.n
