"""The host-buffer entry point on either side of the sizes where the kernels take over from the copy engine, with pinned,
pageable and oddly aligned buffers: the result is that of the device-buffer call, bit for bit, and nothing beside y is written."""
import pytest
import torch

from paper_2512_24545_b200 import inputs, mdbf as M
from helpers import GpuLayer, TORCH_DT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_24545_b200 import build
    build.build()
    assert torch.cuda.is_available()


# bytes of x and of y (bf16): below, at and above 20 KB / 1 MB for x and 256 KB for y
@pytest.mark.parametrize("d_out,d_in,T", [(64, 128, 1), (1000, 10240, 1), (1000, 10248, 1), (8192, 64, 16), (8200, 64, 16), (96, 8192, 64),
                                          (96, 8200, 64), (70, 1001, 31),
                                          (1024, 640, 100), (1280, 12800, 90), (200, 1001, 130)])      # more than 64 tokens: whole, split, expanded order
@pytest.mark.parametrize("memory", ["pinned", "pageable", "pinned_odd"])
def test_host_buffers(d_out, d_in, T, memory):
    host_against_device(inputs.scaled(inputs.qproj(1664), name="host", d_out=d_out, d_in=d_in, k=96, l=4, seed=31), T, memory)


@pytest.mark.parametrize("T", [3, 70])
@pytest.mark.parametrize("memory", ["pinned", "pageable"])
def test_host_buffers_fp32(T, memory):
    host_against_device(inputs.tiny(), T, memory)


def host_against_device(spec, T, memory):
    d_out, d_in, dt = spec.d_out, spec.d_in, TORCH_DT[spec.act_dtype]
    act = M.DTYPES[spec.act_dtype]
    x = torch.from_numpy(inputs.make_activations(spec, T)).to(dt)
    st = torch.cuda.current_stream().cuda_stream

    def host(n):
        off = 1 if memory == "pinned_odd" else 0                  # two bytes past a 16-byte boundary
        buf = torch.full((n + 16 + off,), 7.0, dtype=dt)
        buf = buf if memory == "pageable" else buf.pin_memory()
        return buf, buf[off:off + n]

    with GpuLayer(spec, T) as g:
        xd, yd = x.cuda(), torch.zeros((T, d_out), dtype=dt, device="cuda")
        M.mdbf_linear_forward(g.h, xd.data_ptr(), yd.data_ptr(), T, act, st)
        M.mdbf_prepare_host_staging(g.h)
        _, xh = host(T * d_in)
        xh.copy_(x.reshape(-1))
        whole, yh = host(T * d_out)
        for _ in range(2):
            yh.fill_(3.0)
            M.mdbf_linear_forward_host(g.h, xh.data_ptr(), yh.data_ptr(), T, act, st)
            assert torch.equal(yh.view(T, d_out), yd.cpu())
        assert bool((whole[yh.storage_offset() + T * d_out:] == 7.0).all())
        xh.copy_((x * 2).reshape(-1))                             # other contents of the same buffer
        xd.mul_(2)
        M.mdbf_linear_forward(g.h, xd.data_ptr(), yd.data_ptr(), T, act, st)
        M.mdbf_linear_forward_host_async(g.h, xh.data_ptr(), yh.data_ptr(), T, act, st)
        torch.cuda.synchronize()
        assert torch.equal(yh.view(T, d_out), yd.cpu())
        assert M.mdbf_poll_status(g.h) == 0


@pytest.mark.parametrize("off", [1, 3])
def test_output_off_its_element_boundary(off):
    """y_host anywhere in a pinned byte arena: the copy takes it there."""
    spec = inputs.scaled(inputs.qproj(1664), name="odd", d_out=1000, d_in=640, k=96, l=4, seed=32)
    x = torch.from_numpy(inputs.make_activations(spec, 3)).to(torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream
    with GpuLayer(spec, 3) as g:
        M.mdbf_prepare_host_staging(g.h)
        xh, want = x.pin_memory(), torch.zeros((3, 1000), dtype=torch.bfloat16).pin_memory()
        M.mdbf_linear_forward_host(g.h, xh.data_ptr(), want.data_ptr(), 3, M.BF16, st)
        arena = torch.zeros(6000 + 16, dtype=torch.uint8).pin_memory()
        M.mdbf_linear_forward_host(g.h, xh.data_ptr(), arena.data_ptr() + off, 3, M.BF16, st)
        assert torch.equal(arena[off:off + 6000], want.view(torch.uint8).reshape(-1))
        assert not bool(arena[:off].any()) and not bool(arena[off + 6000:].any())


@pytest.mark.parametrize("mid,T", [(8192, 1), (11008, 1), (4096, 4), (2048, 64)])      # 16, 22, 32 and 256 KB between the layers
@pytest.mark.parametrize("first", ["host_async", "device"])
def test_a_layer_reads_what_the_one_before_it_leaves_in_pinned_memory(mid, T, first):
    """Calls queued on one stream without a wait in between: the second layer's input is the buffer the first one's output goes into."""
    one = inputs.scaled(inputs.qproj(1664), name="one", d_out=mid, d_in=8192, k=2048, l=16, seed=41)
    two = inputs.scaled(inputs.qproj(1664), name="two", d_out=640, d_in=mid, k=256, l=4, seed=42)
    st = torch.cuda.current_stream().cuda_stream
    with GpuLayer(one, T) as a, GpuLayer(two, T) as b:
        M.mdbf_prepare_host_staging(a.h)
        M.mdbf_prepare_host_staging(b.h)
        x = torch.from_numpy(inputs.make_activations(one, T)).to(torch.bfloat16)
        xd, xh = x.cuda(), x.pin_memory()
        buf = torch.zeros((T, mid), dtype=torch.bfloat16).pin_memory()
        out, want = (torch.zeros((T, 640), dtype=torch.bfloat16).pin_memory() for _ in range(2))

        def head():
            if first == "device":
                M.mdbf_linear_forward(a.h, xd.data_ptr(), buf.data_ptr(), T, M.BF16, st)
            else:
                M.mdbf_linear_forward_host_async(a.h, xh.data_ptr(), buf.data_ptr(), T, M.BF16, st)

        head()
        torch.cuda.synchronize()
        M.mdbf_linear_forward_host(b.h, buf.data_ptr(), want.data_ptr(), T, M.BF16, st)
        assert bool(torch.isfinite(want).all()) and float(want.float().abs().max()) > 0
        for _ in range(5):
            buf.zero_()
            out.zero_()
            head()
            M.mdbf_linear_forward_host_async(b.h, buf.data_ptr(), out.data_ptr(), T, M.BF16, st)
            torch.cuda.synchronize()
            assert torch.equal(out, want)
