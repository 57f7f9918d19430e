"""The allocation-free ordering where no cluster can sort the keys (more than 64
cells per axis): a launch pair per digit, none of which waits for another block,
at the edges of the tiles; and the call inside a stream capture."""
import ctypes

import numpy as np
import pytest

from test_gpu_build import keys_of, positions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01341_gb300 import build
    build.build()
    from paper_1807_01341_gb300 import _lib
    return torch, _lib.load()


def order(L, xyz, nc, perm, stream):
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in xyz]
    return L.sph_cell_order_noalloc(*ptr, xyz[0].numel(), 1.0, nc, ctypes.c_void_p(perm.data_ptr()),
                                    ctypes.c_void_p(stream.cuda_stream))


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 8193, 20000, 65535, 65536])
@pytest.mark.parametrize("nc", [65, 255])
def test_order_by_digit_passes(env, n, nc):
    torch, L = env
    pos = positions("clumps" if n % 2 else "uniform", n, nc, np.random.default_rng(n + nc))
    pos[::97] = np.nextafter(1.0, 0.0)  # the largest key
    xyz = [torch.as_tensor(pos[:, k].copy(), device="cuda") for k in range(3)]
    perm = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    assert order(L, xyz, nc, perm, torch.cuda.current_stream()) == 0
    assert np.array_equal(perm.cpu().numpy(), np.argsort(keys_of(pos, nc)[1], kind="stable"))


@pytest.mark.parametrize("nc", [20, 200])
def test_order_inside_a_capture(env, nc):
    torch, L = env
    n = 10000
    rng = np.random.default_rng(nc)
    xyz = [torch.empty(n, dtype=torch.float64, device="cuda").uniform_() for _ in range(3)]
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    assert order(L, xyz, nc, perm, torch.cuda.current_stream()) == 0  # the first call, as documented
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rc = order(L, xyz, nc, perm, torch.cuda.current_stream())
    assert rc == 0
    for _ in range(2):
        pos = rng.uniform(size=(n, 3))
        for k in range(3):
            xyz[k].copy_(torch.as_tensor(pos[:, k].copy()))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(perm.cpu().numpy(), np.argsort(keys_of(pos, nc)[1], kind="stable"))
