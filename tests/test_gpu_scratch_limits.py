"""Calls on several ciphertexts when device memory is short: what runs together needs scratch for all
of them, and where the device has less, the call runs on smaller groups with the same results.  Each
test holds all memory but a slack that suffices for one ciphertext after the other (measured: a half
more than that takes) and not for all at once."""
import numpy as np
import pytest

from paper_2104_09583_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

MB = 1 << 20


class Held:
    """All free device memory but `slack` MB, held while the block runs."""

    def __init__(self, slack):
        self.slack = slack

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.blocks = []
        left, size = torch.cuda.mem_get_info()[0] - self.slack * MB, 1 << 38
        while size >= 2 * MB:
            if size <= left:
                try:
                    self.blocks.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
                    left -= size
                    continue
                except torch.OutOfMemoryError:
                    pass
            size //= 2

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        self.blocks.clear()
        torch.cuda.empty_cache()


def infer_in(slack, log_n, dnum, forest, nf, g):
    """Inference of four full query ciphertexts with `slack` MB free beside the queries and the
    model: its labels and ciphertexts are those of a call with all memory."""
    L, p, n_ct = 10, 8, 4
    ctx = K.copse_ctx_create(log_n, 55, L, dnum)
    made = []
    try:
        model = K.copse_compile_forest(forest, p, nf, log_n)
        made.append((K.copse_model_destroy, model))
        K.copse_model_set_bsgs(model, *g)
        keys, evk = K.copse_keygen(ctx, 7, [model])
        made += [(K.copse_keys_destroy, keys), (K.copse_evk_destroy, evk)]
        i = K.copse_model_info_get(model)
        qs = synth.random_queries(3, n_ct * ((1 << log_n) // (i["block"] * i["n_segments"])), nf, p)
        # one ciphertext first: the model's plaintexts are resident from here on
        none = K.copse_encrypt_features(ctx, keys, model, np.zeros((0, nf), np.uint32), 1)
        made.append((K.copse_ctbuf_destroy, none))
        made.append((K.copse_ctbuf_destroy, K.copse_infer(ctx, evk, model, none)))
        feats = K.copse_encrypt_features(ctx, keys, model, qs, 2)
        made.append((K.copse_ctbuf_destroy, feats))
        assert K.copse_ctbuf_count(feats) == n_ct * p
        with Held(slack):
            res = K.copse_infer(ctx, evk, model, feats)
            made.append((K.copse_ctbuf_destroy, res))
        assert np.array_equal(K.copse_decrypt_labels(ctx, keys, model, res, len(qs)), K.copse_classify_plain(model, qs))
        again = K.copse_infer(ctx, evk, model, feats)
        made.append((K.copse_ctbuf_destroy, again))
        for c in range(n_ct):
            assert np.array_equal(K.copse_ctbuf_export(ctx, res, c, 1 << log_n), K.copse_ctbuf_export(ctx, again, c, 1 << log_n))
    finally:
        for destroy, h in reversed(made):
            destroy(h)
        K.copse_ctx_destroy(ctx)


def test_matrix_products_of_several_query_ciphertexts():
    """N = 2^15: one after the other the four take 0.6 GB, together 2 GB."""
    infer_in(900, 15, 2, synth.random_forest(5, 16, 6, 16, 8, 3), 16, (64, 64))


def test_transforms_without_room_for_the_partial_transform():
    """N = 2^14: with scratch for the tiled transforms' partial results 0.69 GB, in clusters, which
    need none, 0.54 GB."""
    infer_in(600, 14, 3, synth.random_forest(5, 4, 5, 8, 8, 3, complete=False), 8, (32, 32))


def codec(log_n, n_ct, body):
    """body(ctx, keys, model, queries) with a small model and n_ct full query ciphertexts."""
    L, p, nf = 10, 8, 4
    ctx = K.copse_ctx_create(log_n, 55, L, 3)
    made = []
    try:
        model = K.copse_compile_forest(synth.random_forest(5, 2, 4, nf, p, 3, complete=False), p, nf, log_n)
        made.append((K.copse_model_destroy, model))
        keys, evk = K.copse_keygen(ctx, 7, [model])
        made += [(K.copse_keys_destroy, keys), (K.copse_evk_destroy, evk)]
        i = K.copse_model_info_get(model)
        body(ctx, keys, model, synth.random_queries(3, n_ct * ((1 << log_n) // i["block"]), nf, p), made)
    finally:
        for destroy, h in reversed(made):
            destroy(h)
        K.copse_ctx_destroy(ctx)


def test_encryption_of_several_query_ciphertexts():
    """Eight query ciphertexts of eight planes at N = 2^15 (0.32 GB): all samples at once 0.76 GB."""
    def body(ctx, keys, model, qs, made):
        with Held(550):
            few = K.copse_encrypt_features(ctx, keys, model, qs, 2)
            made.append((K.copse_ctbuf_destroy, few))
        all_ = K.copse_encrypt_features(ctx, keys, model, qs, 2)
        made.append((K.copse_ctbuf_destroy, all_))
        assert K.copse_ctbuf_count(few) == K.copse_ctbuf_count(all_) == 64
        for i in range(64):
            assert np.array_equal(K.copse_ctbuf_export(ctx, few, i, 1 << 15), K.copse_ctbuf_export(ctx, all_, i, 1 << 15)), i

    codec(15, 8, body)


def test_decryption_of_several_ciphertexts():
    """Forty ciphertexts of ten primes at N = 2^15: switched down together 0.6 GB, one after the other
    less than what is always left.  They come from another context, whose idle memory is gone."""
    cts = []

    def encrypt(ctx, keys, model, qs, made):
        planes = K.copse_encrypt_features(ctx, keys, model, qs, 2)
        made.append((K.copse_ctbuf_destroy, planes))
        cts.extend(K.copse_ctbuf_export(ctx, planes, i, 1 << 15) for i in range(K.copse_ctbuf_count(planes)))

    def decrypt(ctx, keys, model, qs, made):
        buf = K.copse_ctbuf_import(ctx, np.stack(cts))
        made.append((K.copse_ctbuf_destroy, buf))
        nq = 8 * len(qs)  # eight planes a query ciphertext, each read as a result
        with Held(300):
            few = K.copse_decrypt_labels(ctx, keys, model, buf, nq)
        assert few.any() and (few <= 1).all()
        assert np.array_equal(few, K.copse_decrypt_labels(ctx, keys, model, buf, nq))

    codec(15, 5, encrypt)
    assert len(cts) == 40
    codec(15, 5, decrypt)
