"""The scratch that convolution calls keep between them is bounded and given back."""
import threading

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_scratch_is_bounded_and_given_back():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import unet as N
    x = torch.randn((8, 64, 64, 128, 64), device="cuda").mul_(0.1)    # 8 x 128x64x64 cells: 0.5 GiB converted
    w = torch.randn((64, 64, 27), device="cuda").mul_(0.05)
    y = torch.empty_like(x)
    gw = torch.empty_like(w)
    small = x[:1, :4, :4, :8].contiguous()
    out = torch.empty_like(small)
    N.conv3_forward(small, w, out)                                    # the kernels are loaded
    N.conv3_backward_weights(small, small, gw)
    N.conv3_trim()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    N.conv3_forward(x, w, y)
    N.conv3_backward_weights(x, y, gw)                                # two operands: over 1 GiB
    ref = gw.clone()
    torch.cuda.synchronize()
    kept = free - torch.cuda.mem_get_info()[0]
    N.conv3_trim()
    left = free - torch.cuda.mem_get_info()[0]
    print(f"kept {kept / 2 ** 20:.0f} MiB, after the trim {left / 2 ** 20:.0f} MiB")
    assert kept <= 2 ** 30 + 64 * 2 ** 20 and left <= 64 * 2 ** 20    # a few allocation granules of 2 to 32 MiB
    N.conv3_backward_weights(x, y, gw)                                # and the next call works
    K = x.numel() // 64
    assert (gw - ref).abs().max() <= 8 * K ** 0.5 * 2.0 ** -24 * ref.abs().max()


def test_trims_beside_calls_of_other_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import unet as N
    x = torch.randn((4, 8, 8, 16, 64), device="cuda")
    w = torch.randn((96, 64, 27), device="cuda")
    ref = torch.empty((4, 8, 8, 16, 96), device="cuda")
    N.conv3_forward(x, w, ref)
    bad = []

    def work():
        s = torch.cuda.Stream()
        y = torch.full_like(ref, float("nan"))
        s.wait_stream(torch.cuda.default_stream())
        for _ in range(50):
            N.conv3_forward(x, w, y, s.cuda_stream)
        s.synchronize()
        if not torch.equal(y, ref):
            bad.append(1)

    th = [threading.Thread(target=work) for _ in range(3)]
    for t in th:
        t.start()
    for _ in range(50):
        N.conv3_trim()
    for t in th:
        t.join()
    torch.cuda.synchronize()
    assert not bad
