"""The host-buffer entry point on either side of the sizes where the kernels take over from the copy engine, with pinned,
pageable and oddly aligned buffers: the result is that of the device-buffer call, bit for bit, and nothing beside y is written."""
import pytest
import torch

from paper_2512_24545_b200 import inputs, mdbf as M
from helpers import GpuLayer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_24545_b200 import build
    build.build()
    assert torch.cuda.is_available()


# bytes of x and of y (bf16): below, at and above 20 KB / 1 MB for x and 256 KB for y
@pytest.mark.parametrize("d_out,d_in,T", [(64, 128, 1), (1000, 10240, 1), (1000, 10248, 1), (8192, 64, 16), (8200, 64, 16), (96, 8192, 64),
                                          (96, 8200, 64), (70, 1001, 31)])
@pytest.mark.parametrize("memory", ["pinned", "pageable", "pinned_odd"])
def test_host_buffers(d_out, d_in, T, memory):
    spec = inputs.scaled(inputs.qproj(1664), name="host", d_out=d_out, d_in=d_in, k=96, l=4, seed=31)
    x = torch.from_numpy(inputs.make_activations(spec, T)).to(torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream

    def host(n):
        off = 1 if memory == "pinned_odd" else 0                  # two bytes past a 16-byte boundary
        buf = torch.full((n + 16 + off,), 7.0, dtype=torch.bfloat16)
        buf = buf if memory == "pageable" else buf.pin_memory()
        return buf, buf[off:off + n]

    with GpuLayer(spec, T) as g:
        xd, yd = x.cuda(), torch.zeros((T, d_out), dtype=torch.bfloat16, device="cuda")
        M.mdbf_linear_forward(g.h, xd.data_ptr(), yd.data_ptr(), T, M.BF16, st)
        M.mdbf_prepare_host_staging(g.h)
        _, xh = host(T * d_in)
        xh.copy_(x.reshape(-1))
        whole, yh = host(T * d_out)
        for _ in range(2):
            yh.fill_(3.0)
            M.mdbf_linear_forward_host(g.h, xh.data_ptr(), yh.data_ptr(), T, M.BF16, st)
            assert torch.equal(yh.view(T, d_out), yd.cpu())
        assert bool((whole[yh.storage_offset() + T * d_out:] == 7.0).all())
        xh.copy_((x * 2).reshape(-1))                             # other contents of the same buffer
        xd.mul_(2)
        M.mdbf_linear_forward(g.h, xd.data_ptr(), yd.data_ptr(), T, M.BF16, st)
        M.mdbf_linear_forward_host_async(g.h, xh.data_ptr(), yh.data_ptr(), T, M.BF16, st)
        torch.cuda.synchronize()
        assert torch.equal(yh.view(T, d_out), yd.cpu())
        assert M.mdbf_poll_status(g.h) == 0
