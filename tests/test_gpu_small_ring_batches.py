"""Transforms of N = 2^8, two to a block: batches of odd and even numbers of residue polynomials, with
the words behind the batch left as they are, against the same polynomials one at a time (which the
oracle pins in test_gpu_transforms), and key switches whose digits' own residues (copied, not
transformed) fall on either half of a block, against the oracle (tolerance zero)."""
import numpy as np
import pytest

from oracle import bgv as B
from paper_2104_09583_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import assert_same  # noqa: E402


@pytest.mark.parametrize("log_n", [8, 9])
@pytest.mark.parametrize("polys,nres", [(1, 1), (1, 2), (1, 3), (3, 1), (2, 3), (5, 3), (33, 5), (683, 3)])
def test_batches_equal_single_transforms(log_n, polys, nres):
    N = 1 << log_n
    ctx = K.copse_ctx_create(log_n, 55, 5, 3)
    try:
        pr = np.array(K.copse_ctx_primes(ctx)[:nres], np.uint64)
        rng = np.random.default_rng(polys)
        x = rng.integers(0, 1 << 62, size=(polys, nres, N), dtype=np.uint64) % pr[None, :, None]
        behind = np.full(4 * N, 0x5A5A5A5A5A5A5A5A, np.uint64)
        for inverse in (False, True):
            d = torch.from_numpy(np.concatenate([x.reshape(-1), behind]).view(np.int64)).cuda()
            K.copse_ntt(ctx, d.data_ptr(), polys, nres, inverse=inverse)
            torch.cuda.synchronize()
            got = d.cpu().numpy().view(np.uint64)
            assert (got[polys * nres * N:] == behind).all()
            got = got[:polys * nres * N].reshape(x.shape)
            some = sorted({0, 1, polys // 2, polys - 2, polys - 1} & set(range(polys)))
            for i in some:
                one = torch.from_numpy(x[i].copy().view(np.int64)).cuda()
                K.copse_ntt(ctx, one.data_ptr(), 1, nres, inverse=inverse)
                torch.cuda.synchronize()
                assert_same(got[i], one.cpu().numpy().view(np.uint64), f"polynomial {i}")
            d = torch.from_numpy(got.copy().view(np.int64)).cuda()
            K.copse_ntt(ctx, d.data_ptr(), polys, nres, inverse=not inverse)
            torch.cuda.synchronize()
            assert_same(d.cpu().numpy().view(np.uint64), x, "there and back")
    finally:
        K.copse_ctx_destroy(ctx)


@pytest.mark.parametrize("L,dnum", [(4, 2), (5, 2), (5, 3), (6, 3), (7, 7)])
def test_digits_on_either_half(L, dnum):
    N = 256
    P = B.Params(logN=8, L=L, bits=55, dnum=dnum)
    bgv = B.Bgv(P)
    ctx = K.copse_ctx_create(8, 55, L, dnum)
    try:
        model = K.copse_compile_forest(synth.random_forest(3, 1, 2, 2, 2, 2), 2, 2, 8)
        rot = K.copse_model_rotations(model)[0][-1]
        g = B.galois_rot(8, rot)
        keys, evk = K.copse_keygen(ctx, 21, [model])
        okeys = bgv.keygen(21, [g])
        rng = np.random.default_rng(L)
        cts = [bgv.encrypt_slots(okeys.pk, rng.integers(0, 2, size=N), 8, i) for i in range(2)]
        buf = K.copse_ctbuf_import(ctx, np.stack(cts))
        for h, want in ((K.copse_ct_rotate(ctx, evk, buf, 0, rot), bgv.rotate(cts[0], g, okeys.gk[g])),
                        (K.copse_ct_mul(ctx, evk, buf, 0, buf, 1), bgv.mul(cts[0], cts[1], okeys.rlk))):
            assert_same(K.copse_ctbuf_export(ctx, h, 0, N), want, f"L {L}, dnum {dnum}")
            K.copse_ctbuf_destroy(h)
        K.copse_ctbuf_destroy(buf)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)
