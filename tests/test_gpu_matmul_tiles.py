"""The diagonal products of a plaintext model (csrc/ring.cu) at the edges of their tiles, against
the oracle coefficient for coefficient (tolerance zero: exact modular arithmetic): one
accumulator (the key switch inline), two, three, four and more with a remainder, more than 32 (two
launches), rotations in one chunk of 64 and in several, fewer than a thread keeps in flight, and
partial sums over rotation ranges."""
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

FOREST = (92, 8, 4, 4, 3, 3)  # seed, trees, depth, features, precision, classes
LOG_N = 10


@pytest.mark.parametrize("g", [(0, 0), (90, 70), (60, 40), (40, 64), (4, 9), (64, 16), (2, 3), (3, 2), (66, 67),
                               (27, 17), (22, 14)])
def test_diagonal_products_match_the_oracle(g):
    seed, nt, dp, nf, p, nc = FOREST
    text = synth.random_forest(seed, nt, dp, nf, p, nc, complete=True)
    N = 1 << LOG_N
    om = Cp.compile_forest(text, p, nf, slots_per_row=N // 2)
    assert om.n_seg == 1 and om.q > 128 and om.b > 64
    om_p = B.Params(logN=LOG_N, L=Cp.levels_needed(om) + 1, bits=55, dnum=2)
    qs = synth.random_queries(5, 1, nf, p)
    ctx = K.copse_ctx_create(LOG_N, 55, om_p.L, 2)
    try:
        model = K.copse_compile_forest(text, p, nf, LOG_N)
        K.copse_model_set_bsgs(model, *g)
        keys, evk = K.copse_keygen(ctx, 11, [model])
        feats = K.copse_encrypt_features(ctx, keys, model, qs, 12)
        res = K.copse_infer(ctx, evk, model, feats)
        got = K.copse_ctbuf_export(ctx, res, 0, N)
        for h in (res, feats):
            K.copse_ctbuf_destroy(h)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)
    bgv = B.Bgv(om_p)
    okeys = bgv.keygen(11, Cp.galois_elements(om, LOG_N, g))
    want = Cp.infer(Cp.BgvEngine(bgv, okeys), om, Cp.encrypt_queries(bgv, okeys, om, qs, 12), N, g)
    assert_same(got, want, f"plan {g}")


@pytest.mark.parametrize("g", [(0, 0), (4, 4), (0, 4)])
@pytest.mark.parametrize("nct,fused", [(2, False), (3, True), (9, False)])
def test_ciphertexts_together_match_each_alone(g, nct, fused):
    """The matrix products of several query ciphertexts in one launch (nine: two groups) give each
    ciphertext's own result, word for word."""
    W = synth.WORKLOADS["toy-n1024"]
    N = 1 << W.log_n
    ctx = K.copse_ctx_create(W.log_n, W.bits, W.primes, W.dnum)
    try:
        p, nf = W.precision(), W.n_features()
        model = K.copse_compile_forest(W.forest_texts()[0], p, nf, W.log_n)
        K.copse_model_set_bsgs(model, *g)
        if fused:
            K.copse_model_set_fused(model, True)
        keys, evk = K.copse_keygen(ctx, 7, [model])
        n = 32 * (nct - 1) + 5
        feats = K.copse_encrypt_features(ctx, keys, model, synth.random_queries(n, n, nf, p), 9)
        assert K.copse_ctbuf_count(feats) == nct * p
        res = K.copse_infer(ctx, evk, model, feats)
        for q in range(nct):
            one = K.copse_ctbuf_import(ctx, np.stack([K.copse_ctbuf_export(ctx, feats, q * p + i, N) for i in range(p)]))
            alone = K.copse_infer(ctx, evk, model, one)
            assert_same(K.copse_ctbuf_export(ctx, res, q, N), K.copse_ctbuf_export(ctx, alone, 0, N), f"ciphertext {q}")
            K.copse_ctbuf_destroy(alone)
            K.copse_ctbuf_destroy(one)
        for h in (res, feats):
            K.copse_ctbuf_destroy(h)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)
