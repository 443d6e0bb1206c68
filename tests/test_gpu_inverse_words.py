"""The inverse transform of the rings below 2^12 takes words of [0, 2q) (a lazily added residue need
not be corrected before it): the result is that of the residues, word for word, and its forward
transform gives the residues back."""
import numpy as np
import pytest

from oracle import bgv as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import assert_same  # noqa: E402


@pytest.mark.parametrize("bits", [36, 55])
@pytest.mark.parametrize("log_n", [4, 7, 8, 9, 10, 11])
def test_inverse_of_words_below_two_q(log_n, bits):
    L, N = 2, 1 << log_n
    P = B.Params(logN=log_n, L=L, bits=bits, dnum=2)
    ctx = K.copse_ctx_create(log_n, bits, L, 2)
    try:
        rng = np.random.default_rng(log_n)
        x = np.empty((4, L, N), np.uint64)
        raised = np.zeros((4, N), bool)
        raised[0, ::3] = True
        raised[1, 1::2] = True
        raised[2] = True
        raised[3, N // 2:] = True
        for r, q in enumerate(P.q):
            x[:3, r] = rng.integers(0, q, size=(3, N), dtype=np.uint64)
            x[3, r] = np.where(raised[3], q - 1, 0)  # 0 and the largest word, 2q - 1
        y = x + raised[:, None, :] * np.array(P.q, np.uint64)[None, :, None]
        a, b = (torch.from_numpy(z.view(np.int64)).cuda() for z in (x, y))
        for d in (a, b):
            K.copse_ntt(ctx, d.data_ptr(), 4, L, inverse=True)
        torch.cuda.synchronize()
        got = b.cpu().numpy().view(np.uint64)
        assert_same(got, a.cpu().numpy().view(np.uint64), "words raised by q")
        # and forward again: the residues
        K.copse_ntt(ctx, b.data_ptr(), 4, L)
        torch.cuda.synchronize()
        assert_same(b.cpu().numpy().view(np.uint64), x, "forward of the inverse")
    finally:
        K.copse_ctx_destroy(ctx)
