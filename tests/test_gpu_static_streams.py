"""Calls of the allocation-free step share no state: steps of different
buffers enqueued on two streams, nothing ordering them, have the bits of the
same steps one after the other."""
import numpy as np
import pytest

from helpers import lbm_mod

pytestmark = pytest.mark.gpu

# the two forms of the step (a cube, and rows of three cells), and D2Q9
CASES = [("D3Q19", (61, 50, 47)), ("D3Q19", (3, 200, 240)), ("D2Q9", (301, 405, 1))]


@pytest.mark.parametrize("a", CASES)
@pytest.mark.parametrize("b", CASES)
def test_two_streams(a, b):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    lbm = lbm_mod()

    def buffers(lat, ext, seed):
        q = 19 if lat == "D3Q19" else 9
        f = np.random.default_rng(seed).uniform(0.05, 0.15, size=q * int(np.prod(ext)))
        x = torch.from_numpy(f.astype(np.float32)).cuda()
        return x, torch.empty_like(x)

    def step(lat, ext, x, y, stream):
        lbm.step_static_f32(lat, *ext, 0.9, -5.0, 1.0, x.data_ptr(), y.data_ptr(),
                            stream.cuda_stream)

    def run(streams):
        bufs = [buffers(*a, 1), buffers(*b, 2)]
        torch.cuda.synchronize()
        for _ in range(12):
            for k, case in enumerate((a, b)):
                step(*case, *bufs[k], streams[k])
                bufs[k] = bufs[k][::-1]
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x, _ in bufs]

    one = torch.cuda.Stream()
    want = run([one, one])
    got = run([torch.cuda.Stream(), torch.cuda.Stream()])
    for g, w in zip(got, want):
        assert np.isfinite(w).all() and (g == w).all()
