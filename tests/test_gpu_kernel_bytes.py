"""The kernel timers' algorithmic bytes of the diagonal products: query ciphertexts that run together
account for what as many single ones do (one accumulator: one launch each, its own sums only), and a
first launch writes its sums without reading them."""
import pytest

from paper_2104_09583_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def test_one_accumulator_several_lanes():
    """Three trees of depth 1: the reshuffle and the level product have one accumulator each."""
    log_n, L, dnum, p, nf = 9, 8, 4, 2, 2
    N, alpha = 1 << log_n, 2
    ctx = K.copse_ctx_create(log_n, 50, L, dnum)
    made = []
    try:
        model = K.copse_compile_forest(synth.random_forest(4, 3, 1, nf, p, 2), p, nf, log_n)
        made.append((K.copse_model_destroy, model))
        keys, evk = K.copse_keygen(ctx, 3, [model])
        made += [(K.copse_keys_destroy, keys), (K.copse_evk_destroy, evk)]
        i = K.copse_model_info_get(model)
        assert i["depth"] == 1 and i["n_segments"] == 1 and i["n_rot_reshuffle"] > 0 and i["n_rot_level"] > 0
        got = {}
        for n_ct in (1, 3):
            qs = synth.random_queries(5, n_ct * (N // i["block"]), nf, p)
            feats = K.copse_encrypt_features(ctx, keys, model, qs, 9)
            made.append((K.copse_ctbuf_destroy, feats))
            made.append((K.copse_ctbuf_destroy, K.copse_infer(ctx, evk, model, feats)))  # the model is resident
            K.copse_stats_reset()
            K.copse_stats_enable(True)
            made.append((K.copse_ctbuf_destroy, K.copse_infer(ctx, evk, model, feats)))
            K.copse_stats_enable(False)
            got[n_ct] = K.copse_stats_get("mm_fused")
        assert got[1]["launches"] == 2 and got[3]["launches"] == 6
        assert got[3]["bytes"] == 3 * got[1]["bytes"]
        # levels: one prime each for the comparison leaves, the combine product and the reshuffle
        want = 0
        for ell, nr in ((L - 2, i["n_rot_reshuffle"]), (L - 3, i["n_rot_level"])):
            nx, nd = ell + alpha, -(-ell // alpha)
            want += 8 * N * (nr * nx + 2 * nx + nr * 2 * nd * nx + nd * nx + ell)
        assert got[1]["bytes"] == want
    finally:
        K.copse_stats_enable(False)
        K.copse_stats_reset()
        for destroy, h in reversed(made):
            destroy(h)
        K.copse_ctx_destroy(ctx)
