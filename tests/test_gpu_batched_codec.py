"""Encryption and decryption of several query ciphertexts at once (csrc/ring.cu): ciphertexts beyond
the first group that fits the samples' scratch, a last one part full, and none, against the oracle
plane for plane (tolerance zero) and through the bits of a result."""
import numpy as np
import pytest

from oracle import bgv as B
from oracle import copse as Cp
from paper_2104_09583_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import assert_same  # noqa: E402


def test_planes_beyond_the_first_group():
    """N = 2^15, 16 primes, 16 planes: five ciphertexts' samples fit 1 GB, so seven make two groups."""
    log_n, L, p, nf = 15, 16, 16, 3
    text = synth.random_forest(5, 1, 2, nf, p, 2)
    P = B.Params(logN=log_n, L=L, bits=55, dnum=3)
    om = Cp.compile_forest(text, p, nf)
    per_ct = P.N // om.block
    n = 6 * per_ct + 5
    qs = synth.random_queries(77, n, nf, p)
    bgv = B.Bgv(P)
    okeys = bgv.keygen(4, [])
    ctx = K.copse_ctx_create(log_n, 55, L, 3)
    try:
        model = K.copse_compile_forest(text, p, nf, log_n)
        keys, evk = K.copse_keygen(ctx, 4, [])
        buf = K.copse_encrypt_features(ctx, keys, model, qs, 31)
        assert K.copse_ctbuf_count(buf) == 7 * p
        for c, planes in ((0, (0,)), (4, (15,)), (5, (0, 7)), (6, (15,))):
            bits = Cp.feature_planes(om, qs[c * per_ct:(c + 1) * per_ct], P.N)
            for i in planes:
                want = bgv.encrypt_slots(okeys.pk, bits[i], 31, c * p + i)
                assert_same(K.copse_ctbuf_export(ctx, buf, c * p + i, P.N), want, f"ciphertext {c}, plane {i}")
        K.copse_ctbuf_destroy(buf)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)


@pytest.mark.parametrize("n", [0, 1, 33, 70])
def test_bits_of_several_results(n):
    """Inference and decryption of up to three query ciphertexts of 32 queries, the last part full."""
    W = synth.WORKLOADS["toy-n1024"]
    text = W.forest_texts()[0]
    ctx = K.copse_ctx_create(W.log_n, W.bits, W.primes, W.dnum)
    try:
        model = K.copse_compile_forest(text, W.precision(), W.n_features(), W.log_n)
        keys, evk = K.copse_keygen(ctx, 7, [model])
        qs = synth.random_queries(n, n, W.n_features(), W.precision())
        feats = K.copse_encrypt_features(ctx, keys, model, qs, 3)
        res = K.copse_infer(ctx, evk, model, feats)
        bits = K.copse_decrypt_labels(ctx, keys, model, res, n)
        assert np.array_equal(bits, K.copse_classify_plain(model, qs))
        for h in (feats, res):
            K.copse_ctbuf_destroy(h)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)
