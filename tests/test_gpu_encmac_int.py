"""The integer multiply-accumulate of the encrypted model (csrc/encmac_int.cu) and its
tensor-core form (csrc/encmac.cu), each fixed in turn, on the sizes at the edges of the integer
kernel's tiles: one, two and three query ciphertexts (one or two per thread), 17 (two tiles), odd
accumulator counts, baby steps below, at and above its chunk of 32, an absent diagonal in the
last giant step, and the largest 55-bit primes.  Every result equals the oracle's residue for
residue (tolerance zero: exact modular arithmetic), and the two kernels' results are equal."""
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

FOREST = (71, 2, 3, 3, 3, 3)  # seed, trees, depth, features, precision, classes
LOG_N = 8


@pytest.mark.parametrize("g,n_ct", [((0, 0), 1), ((5, 3), 2), ((5, 3), 3), ((7, 14), 17), ((32, 1), 2), ((1, 5), 5)])
def test_both_kernels_match_the_oracle(g, n_ct):
    seed, nt, dp, nf, p, nc = FOREST
    text = synth.random_forest(seed, nt, dp, nf, p, nc, complete=True)
    N = 1 << LOG_N
    om = Cp.compile_forest(text, p, nf, slots_per_row=N // 2)
    L = Cp.levels_needed(om) + 1
    per_ct = N // (om.block * om.n_seg)
    qs = synth.random_queries(31 + n_ct, n_ct * per_ct, nf, p)
    ctx = K.copse_ctx_create(LOG_N, 55, L, 3)
    got = {}
    try:
        model = K.copse_compile_forest(text, p, nf, LOG_N)
        K.copse_model_set_encrypted(model, True)
        K.copse_model_set_bsgs(model, *g)
        keys, evk = K.copse_keygen(ctx, 57, [model])
        K.copse_encrypt_model(ctx, keys, model, 2468)
        feats = K.copse_encrypt_features(ctx, keys, model, qs, 35)
        for kernel in ("tensor", "integer"):
            K.copse_ctx_set_enc_mac(ctx, kernel)
            res = K.copse_infer(ctx, evk, model, feats)
            assert K.copse_ctx_device_status(ctx) == 0
            got[kernel] = [K.copse_ctbuf_export(ctx, res, c, N) for c in range(n_ct)]
            K.copse_ctbuf_destroy(res)
        with pytest.raises(K.CopseError):
            K._check(K.library().copse_ctx_set_enc_mac(ctx, 3))
        K.copse_ctbuf_destroy(feats)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
    finally:
        K.copse_ctx_destroy(ctx)
    for c in range(n_ct):
        assert np.array_equal(got["tensor"][c], got["integer"][c]), f"query ciphertext {c}"
    P = B.Params(logN=LOG_N, L=L, bits=55, dnum=3)
    bgv = B.Bgv(P)
    rs, ls = Cp.encrypted_rotation_sets(om, g)
    okeys = bgv.keygen(57, sorted(set(B.galois_rot(LOG_N, k) for k in rs + ls)))
    em = Cp.encrypt_model(bgv, okeys.sk, om, N, 2468, g)
    E = Cp.BgvEngine(bgv, okeys, encrypted_model=True, enc_model=em)
    for c in sorted({0, n_ct // 2, n_ct - 1}):
        X = Cp.encrypt_queries(bgv, okeys, om, qs[c * per_ct:(c + 1) * per_ct], 35, index0=c * p)
        assert_same(got["integer"][c], Cp.infer(E, om, X, N), f"query ciphertext {c}")
