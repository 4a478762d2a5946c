"""The pixel sort at its edges: list lengths around a round of lanes, a round of the block and
the kernel's register forms, one to four radix passes, lists of one pixel and sorted lists."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def z_keys(pix, width):
    def spread(v):
        v = v.astype(np.uint64)
        return sum(((v >> np.uint64(b)) & np.uint64(1)) << np.uint64(2 * b) for b in range(16))
    return spread(pix % width) | (spread(pix // width) << np.uint64(1))


@pytest.mark.parametrize("size", [(16, 16), (100, 100), (4001, 3001), (65535, 32767)])
@pytest.mark.parametrize("n", [1, 31, 33, 1024, 1025, 2048, 2049, 8192, 8193, 16383])
def test_sort_is_the_z_order(size, n):
    from paper_2509_14442_gb300 import bos
    w, h = size
    rng = np.random.default_rng(n + w)
    pix = rng.integers(0, w * h, n).astype(np.int32)
    want = pix[np.argsort(z_keys(pix, w), kind="stable")]
    for case, ref in ((pix, want), (want, want), (want[::-1], want), (np.full(n, pix[0]), np.full(n, pix[0]))):
        t = torch.as_tensor(case.copy(), device="cuda")
        bos.bos_sort_pixels(t.data_ptr(), n, w, h, torch.cuda.current_stream().cuda_stream)
        assert np.array_equal(t.cpu().numpy(), ref)
