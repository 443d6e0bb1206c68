"""The transforms of every ring from N = 2^8 on (each has its own stage counts and tile shapes: one
block below 2^12, else columns and rows in one launch, clusters, and in two, tiled), plain and
fused with the base conversions, against the oracle coefficient for coefficient (tolerance zero):
import and export (plain both ways), a product (ModUp; relinearise and drop), a rotation (ModUp;
ModDown with a permuted addend), a modulus switch, at 55-bit primes and digits of one, two and
three primes, and the negacyclic product of copse_poly_mul."""
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

ALWAYS = 1 << 30


@pytest.mark.parametrize("log_n,dnum", [(8, 3), (9, 5), (10, 2), (11, 3), (12, 5), (12, 2), (13, 3), (14, 2), (15, 3)])
def test_ring_operations_match_the_oracle(log_n, dnum):
    L, N = 5, 1 << log_n
    P = B.Params(logN=log_n, L=L, bits=55, dnum=dnum)
    bgv = B.Bgv(P)
    ctx = K.copse_ctx_create(log_n, 55, L, dnum)
    made = []
    try:
        assert K.copse_ctx_primes(ctx) == P.primes
        model = K.copse_compile_forest(synth.random_forest(3, 1, 2, 2, 2, 2), 2, 2, log_n)
        rot = K.copse_model_rotations(model)[0][-1]
        g = B.galois_rot(log_n, rot)
        keys, evk = K.copse_keygen(ctx, 21, [model])
        okeys = bgv.keygen(21, [g])
        rng = np.random.default_rng(log_n)
        cts = [bgv.encrypt_slots(okeys.pk, rng.integers(0, 2, size=N), 8, i) for i in range(2)]
        want = {"mul": bgv.mul(cts[0], cts[1], okeys.rlk), "rotate": bgv.rotate(cts[0], g, okeys.gk[g]),
                "modswitch": bgv.modswitch(cts[1]), "import/export": cts[0]}
        for most in (ALWAYS, 0):
            K.copse_ctx_set_ntt_cluster_max(ctx, most)
            K.copse_ctx_set_ntt_fused_max(ctx, most)
            buf = K.copse_ctbuf_import(ctx, np.stack(cts))
            got = {"mul": K.copse_ct_mul(ctx, evk, buf, 0, buf, 1), "rotate": K.copse_ct_rotate(ctx, evk, buf, 0, rot),
                   "modswitch": K.copse_ct_modswitch(ctx, buf, 1), "import/export": buf}
            for what, h in got.items():
                assert_same(K.copse_ctbuf_export(ctx, h, 0, N), want[what], f"{what}, {'clusters' if most else 'tiled'}")
                made.append(h)
    finally:
        for h in made:
            K.copse_ctbuf_destroy(h)
        K.copse_keys_destroy(keys)
        K.copse_evk_destroy(evk)
        K.copse_model_destroy(model)
        K.copse_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n", [8, 9, 11, 12, 13])
@pytest.mark.parametrize("most", [ALWAYS, 0])
def test_negacyclic_product_matches_the_oracle(log_n, most):
    P = B.Params(logN=log_n, L=3, bits=55, dnum=3)
    ctx = K.copse_ctx_create(log_n, 55, 3, 3)
    try:
        K.copse_ctx_set_ntt_cluster_max(ctx, most)
        rng = np.random.default_rng(2)
        # the largest residues in front
        a, b = (np.stack([np.concatenate([np.full(8, q - 1, np.uint64), rng.integers(0, q, size=P.N - 8, dtype=np.uint64)])
                          for q in P.q]) for _ in range(2))
        da, db = (torch.from_numpy(x.view(np.int64)).cuda() for x in (a, b))
        dc = torch.empty_like(da)
        K.copse_poly_mul(ctx, da.data_ptr(), db.data_ptr(), dc.data_ptr(), 3)
        torch.cuda.synchronize()
        want = np.zeros_like(a)
        for r, q in enumerate(P.q):
            B.lib().or_negacyclic_mul(np.ascontiguousarray(a[r]), np.ascontiguousarray(b[r]), P.logN, q, want[r])
        assert_same(dc.cpu().numpy().view(np.uint64), want, "negacyclic product")
    finally:
        K.copse_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n,bits", [(8, 36), (11, 36), (12, 36), (13, 36), (14, 40), (15, 40), (8, 55), (11, 55),
                                        (12, 55), (13, 55), (14, 55), (15, 55)])
def test_transforms_at_the_ends_of_their_lazy_ranges(log_n, bits):
    """Forward and inverse of residues all q - 1, all zero but one, alternating 0 and q - 1, and
    random ones, at the smallest and the largest primes, in clusters and tiled."""
    L, N = 2, 1 << log_n
    P = B.Params(logN=log_n, L=L, bits=bits, dnum=2)
    ctx = K.copse_ctx_create(log_n, bits, L, 2)
    try:
        rng = np.random.default_rng(log_n + bits)
        x = np.zeros((4, L, N), np.uint64)
        for r, q in enumerate(P.q):
            x[0, r] = q - 1
            x[1, r, N - 1] = q - 1
            x[2, r, ::2] = q - 1
            x[3, r] = rng.integers(0, q, size=N, dtype=np.uint64)
        for most in (ALWAYS, 0):
            K.copse_ctx_set_ntt_cluster_max(ctx, most)
            d = torch.from_numpy(x.view(np.int64)).cuda()
            K.copse_ntt(ctx, d.data_ptr(), 4, L)
            f = d.clone()
            K.copse_ntt(ctx, d.data_ptr(), 4, L, inverse=True)
            # the inverse of the largest values, forward again
            e = torch.from_numpy(x.view(np.int64)).cuda()
            K.copse_ntt(ctx, e.data_ptr(), 4, L, inverse=True)
            K.copse_ntt(ctx, e.data_ptr(), 4, L)
            torch.cuda.synchronize()
            got = f.cpu().numpy().view(np.uint64)
            assert_same(d.cpu().numpy().view(np.uint64), x, "forward and back")
            assert_same(e.cpu().numpy().view(np.uint64), x, "inverse and forward")
            for r, q in enumerate(P.q):
                assert (got[:, r] < q).all()
                # products of the transforms are the transforms of the products
                out = np.zeros(N, np.uint64)
                B.lib().or_negacyclic_mul(x[0, r].copy(), x[3, r].copy(), log_n, q, out)
                prod = np.array([int(a) * int(b) % q for a, b in zip(got[0, r], got[3, r])], np.uint64)
                t = torch.from_numpy(np.stack([prod] * L).view(np.int64)).cuda()
                K.copse_ntt(ctx, t.data_ptr(), 1, L, inverse=True)
                torch.cuda.synchronize()
                assert_same(t.cpu().numpy().view(np.uint64)[r], out, f"product, prime {r}")
    finally:
        K.copse_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n", [8, 11, 12, 14, 15])
def test_forward_of_words_that_are_not_residues(log_n):
    """The forward transform of x + k q is that of x, up to words of 2^64 - 2^60."""
    L, N = 2, 1 << log_n
    P = B.Params(logN=log_n, L=L, bits=55, dnum=2)
    ctx = K.copse_ctx_create(log_n, 55, L, 2)
    try:
        rng = np.random.default_rng(log_n)
        x = np.stack([rng.integers(0, q, size=N, dtype=np.uint64) for q in P.q])
        for most in (ALWAYS, 0):
            K.copse_ctx_set_ntt_cluster_max(ctx, most)
            for top in (1 << 57, 1 << 61, 1 << 62, 1 << 63, (1 << 64) - (1 << 60)):
                y = x.copy()
                for r, q in enumerate(P.q):
                    y[r, ::3] += np.uint64(top // q - 1) * np.uint64(q)
                a, b = (torch.from_numpy(z.view(np.int64)).cuda() for z in (x, y))
                for d in (a, b):
                    K.copse_ntt(ctx, d.data_ptr(), 1, L)
                torch.cuda.synchronize()
                assert_same(b.cpu().numpy().view(np.uint64), a.cpu().numpy().view(np.uint64), f"words below {top}")
    finally:
        K.copse_ctx_destroy(ctx)
