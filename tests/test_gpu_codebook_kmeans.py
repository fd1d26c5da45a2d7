"""GPU parity of btc_codebook_kmeans against the numpy oracle (bit-exact: integer work)."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

pytestmark = pytest.mark.gpu

import paper_2506_12040_b200 as btc  # noqa: E402
from oracle import codebook_kmeans as km  # noqa: E402


def _vectors(n, v, kind, seed):
    """Seeded +-1 vectors: 'noisy' = a few prototypes with flipped elements (what binarised weight blocks of a
    trained layer look like: a skewed pattern distribution), 'iid' = independent fair signs, 'few' = at most a
    handful of distinct vectors."""
    rng = np.random.default_rng(seed)
    if kind == "iid":
        return np.where(rng.random((n, v)) < 0.5, 1, -1).astype(np.int8)
    protos = np.where(rng.random((7 if kind == "few" else 60, v)) < 0.5, 1, -1).astype(np.int8)
    B = protos[rng.integers(0, protos.shape[0], n)]
    if kind == "noisy":
        B = np.where(rng.random(B.shape) < 0.08, -B, B).astype(np.int8)
    return B


def _run(B, v, Kc, max_iter):
    words = torch.from_numpy(km.pack_words(B).view(np.int32).copy()).cuda()
    C, z, info = btc.codebook_kmeans(words, v, Kc, max_iter)
    torch.cuda.synchronize()
    return C.cpu().numpy().view(np.uint32), z.cpu().numpy().view(np.uint16), info.cpu().numpy()


CASES = [
    # n, v, Kc, max_iter, kind
    (8, 4, 2, 10, "fixture"),
    (5000, 8, 16, 30, "noisy"),
    (20000, 12, 256, 25, "noisy"),
    (30000, 10, 100, 3, "iid"),          # stops by max_iter
    (4000, 16, 300, 12, "noisy"),
    (3000, 16, 64, 40, "iid"),           # nearly all vectors distinct
    (2000, 9, 50, 10, "few"),            # fewer distinct vectors than centroids
    (1, 5, 3, 4, "iid"),
    (70000, 13, 5000, 6, "noisy"),       # ragged: many tiles of centroids and patterns
    (30000, 20, 700, 8, "noisy"),        # the longest vectors of the paper's range
    (9000, 18, 3000, 5, "iid"),
    (100, 1, 2, 3, "iid"),               # one element per vector: two patterns
    (1000, 6, 1, 5, "noisy"),            # a single centroid: the bitwise majority
    (500, 16, 65536, 3, "iid"),          # the largest codebook, far more slots than vectors
]


@pytest.mark.parametrize("n,v,Kc,max_iter,kind", CASES)
def test_kmeans_matches_oracle_bit_for_bit(n, v, Kc, max_iter, kind):
    if kind == "fixture":
        B = np.array([[1, 1, 1, 1]] * 3 + [[-1, 1, 1, 1]] * 2 + [[-1, -1, -1, 1], [-1, -1, -1, -1], [-1, -1, 1, -1]], dtype=np.int8)
    else:
        B = _vectors(n, v, kind, seed=n + v + Kc)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, max_iter, with_flag=True)
    C, z, info = _run(B, v, Kc, max_iter)
    k_eff = min(Kc, n_unique)
    assert info[0] == iters_ref and info[1] == k_eff and info[2] == n_unique
    assert np.array_equal(C[:k_eff], km.pack_words(C_ref)) and not C[k_eff:].any()
    assert np.array_equal(z.astype(np.int64), z_ref)
    assert info[3] == int(converged)


@pytest.mark.parametrize("n,v,Kc,offset", [(300000, 8, 100, 0), (120000, 3, 5, 1), (66000, 16, 2500, 3), (40000, 17, 500, 2),
                                           (5000, 10, 400, 0), (2049, 9, 512, 1)])
def test_kmeans_edges(n, v, Kc, offset):
    """Where the single launch can go wrong: frequencies past the last bin of the frequency histogram, vectors that start
    off a 16-byte boundary with a ragged end, one more and one less bit than a half of the E-step covers, the
    histogram in shared memory (v = 16) and in global memory (v = 17)."""
    B = _vectors(n, v, "noisy", seed=n + v)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, 4, with_flag=True)
    buf = torch.zeros(n + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(km.pack_words(B).view(np.int32).copy()).cuda()
    C, z, info = btc.codebook_kmeans(buf[offset:], v, Kc, 4)
    torch.cuda.synchronize()
    k_eff = min(Kc, n_unique)
    assert info.tolist() == [iters_ref, k_eff, n_unique, int(converged)]
    assert np.array_equal(C.cpu().numpy().view(np.uint32)[:k_eff], km.pack_words(C_ref))
    assert np.array_equal(z.cpu().numpy().view(np.uint16).astype(np.int64), z_ref)
    assert btc.device_status() == 0


@pytest.mark.parametrize("n,v,Kc,kind,repeat,z_off,rounds", [(2000, 12, 20, "iid", 1, 0, 4), (2000, 12, 20, "iid", 1049, 3, 4), (70003, 16, 40, "noisy", 1, 1, 3),
                                                             (6001, 18, 40, "iid", 1, 2, 3), (50001, 2, 3, "noisy", 1, 4, 2)])
def test_kmeans_votes_move_over_rounds(n, v, Kc, kind, repeat, z_off, rounds):
    """Three and four rounds, with votes carried from one to the next in counts of 21 and (from 2^21 vectors on; the same
    vectors over and over have the same result) 32 bits; assignments at every alignment of z; fewer patterns than a
    16-byte piece of the histogram (there no votes move)."""
    B = _vectors(n, v, kind, seed=n + v)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, 6, with_flag=True)
    assert iters_ref == rounds
    B, z_ref, n = np.tile(B, (repeat, 1)), np.tile(z_ref, repeat), n * repeat
    words = torch.from_numpy(km.pack_words(B).view(np.int32).copy()).cuda()
    ws = torch.empty(int(btc.lib.btc_codebook_kmeans_workspace_bytes(v, Kc)), dtype=torch.uint8, device="cuda")
    C, info = torch.empty(Kc, dtype=torch.int32, device="cuda"), torch.empty(4, dtype=torch.int32, device="cuda")
    z = torch.full((n + 8,), -7, dtype=torch.int16, device="cuda")
    assert btc.lib.btc_codebook_kmeans(words.data_ptr(), n, v, Kc, 6, C.data_ptr(), z.data_ptr() + 2 * z_off, info.data_ptr(),
                                       ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    k_eff = min(Kc, n_unique)
    assert info.tolist() == [iters_ref, k_eff, n_unique, int(converged)]
    assert np.array_equal(C.cpu().numpy().view(np.uint32)[:k_eff], km.pack_words(C_ref))
    got = z.cpu().numpy()
    assert np.array_equal(got[z_off:z_off + n].view(np.uint16).astype(np.int64), z_ref)
    assert (got[:z_off] == -7).all() and (got[z_off + n:] == -7).all()


def _pulled_apart(v, Kc, top, seed):
    """Every pattern once; the most frequent ones, the first centroids, side by side, the next most frequent ones spread out: after
    the first round every centroid leaves its place, and most patterns change their cluster."""
    rng = np.random.default_rng(seed)
    cnt = np.ones(1 << v, dtype=np.int64)
    bits = max(Kc - 1, 1).bit_length()
    for j, far in enumerate(rng.integers(0, 1 << (v - bits), Kc)):
        cnt[j] = top + 100
        for q in range(3):
            cnt[((far ^ (1 << q if q else 0)) << bits) | j] = top - q
    return rng.permutation(np.repeat(np.arange(1 << v), cnt))


@pytest.mark.parametrize("v,Kc,top,max_iter,repeat,rounds,least", [(12, 8, 900, 2, 1, 2, 0.5), (14, 16, 900, 25, 1, 5, 0.5), (14, 16, 3000, 3, 25, 3, 0.5), (14, 100, 900, 25, 1, 5, 0.5),
                                                                   (13, 1, 900, 25, 1, 2, 0.0), (16, 5, 900, 4, 1, 4, 0.5)])
def test_kmeans_most_patterns_move(v, Kc, top, max_iter, repeat, rounds, least):
    """Votes in several copies (64 patterns or more per centroid and copy): 8, 16, 16 (counts of 32 bits, and frequencies past the
    last bin, whose list was in the same memory), 2, 32 (more copies than CTAs) and 32 of them; most patterns move in the second
    round, where a run may end."""
    words = _pulled_apart(v, Kc, top, v + Kc)
    B = km.unpack_words(words, v)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, max_iter, with_flag=True)
    assert iters_ref == rounds and n_unique >= 2 * 64 * Kc
    z1, z2 = (km.optimize_codebook(B, Kc, r)[1] for r in (1, 2))
    first = np.unique(words, return_index=True)[1]
    assert (z1[first] != z2[first]).mean() >= least
    C, z, info = _run(np.tile(B, (repeat, 1)), v, Kc, max_iter)
    assert info.tolist() == [iters_ref, Kc, n_unique, int(converged)]
    assert np.array_equal(C, km.pack_words(C_ref)) and np.array_equal(z.astype(np.int64), np.tile(z_ref, repeat))
    assert btc.device_status() == 0


@pytest.mark.parametrize("n,v,Kc,kind", [(6001, 18, 40, "iid"), (6003, 17, 200, "noisy"), (149, 20, 20, "iid")])
def test_kmeans_shares_past_the_end(n, v, Kc, kind):
    """More CTAs than shares of vectors, and a number of vectors that four does not divide: the last ones are counted once."""
    B = _vectors(n, v, kind, seed=n + v)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, 6, with_flag=True)
    C, z, info = _run(B, v, Kc, 6)
    assert info.tolist() == [iters_ref, min(Kc, n_unique), n_unique, int(converged)]
    assert np.array_equal(C[:info[1]], km.pack_words(C_ref)) and np.array_equal(z.astype(np.int64), z_ref)


@pytest.mark.parametrize("n,v,Kc,kind,max_iter", [(1, 5, 3, "iid", 1), (1, 5, 3, "iid", 2), (1, 5, 3, "iid", 3), (2000, 9, 50, "few", 1), (2000, 9, 50, "few", 2),
                                                  (20000, 12, 256, "noisy", 1), (20000, 12, 256, "noisy", 2), (20000, 12, 256, "noisy", 3), (20000, 12, 256, "noisy", 4),
                                                  (300000, 14, 9000, "noisy", 2), (300000, 14, 9000, "noisy", 3)])
def test_kmeans_ends_where_no_centroid_moves(n, v, Kc, kind, max_iter):
    """The last round is only counted where no centroid moved before it: with and without a round left to count, centroids that
    stay from the first round on (as many as patterns) and that move first."""
    B = _vectors(n, v, kind, seed=n + v)
    C_ref, z_ref, iters_ref, n_unique, converged = km.optimize_codebook(B, Kc, max_iter, with_flag=True)
    C, z, info = _run(B, v, Kc, max_iter)
    assert info.tolist() == [iters_ref, min(Kc, n_unique), n_unique, int(converged)]
    assert np.array_equal(C[:info[1]], km.pack_words(C_ref)) and np.array_equal(z.astype(np.int64), z_ref)
    assert btc.device_status() == 0


@pytest.mark.parametrize("v,Kc", [(3, 5), (5, 32), (8, 60), (9, 400)])
def test_kmeans_frequencies_around_the_last_bin(v, Kc):
    """All patterns, at frequencies on both sides of the last bin (2047 and more are ranked pairwise), many of them equal: parts of
    one pattern and of several; where a rank is wrong a centroid is another, or starts in another's place."""
    cnt = np.random.default_rng(v).integers(2041, 2053, 1 << v)
    words = np.random.default_rng(Kc).permutation(np.repeat(np.arange(1 << v, dtype=np.uint32), cnt))
    C_ref, n_unique = km.initial_codebook(km.unpack_words(words, v), Kc)
    C, z, info = (t.cpu().numpy() for t in btc.codebook_kmeans(torch.from_numpy(words.view(np.int32)).cuda(), v, Kc, 1))
    z_pat = km.e_step(km.unpack_words(np.arange(1 << v), v), C_ref)
    assert info.tolist() == [1, Kc, n_unique, 0] and np.array_equal(z.view(np.uint16), z_pat[words])
    U = km.unpack_words(np.arange(1 << v), v).astype(np.int64) * cnt[:, None]
    sums = np.stack([U[z_pat == k].sum(axis=0) for k in range(Kc)])
    assert np.array_equal(C.view(np.uint32), km.pack_words(np.where(sums >= 0, 1, -1)))
    assert btc.device_status() == 0


def test_kmeans_feeds_the_layer():
    """The construction's outputs are the layer's inputs: centroids -> btc_codebook_pack, z -> idx; decoding them
    gives the nearest-centroid approximation of the sign matrix, whose Hamming error equals the oracle's objective."""
    N, K, v, Kc = 64, 256, 16, 128
    B = _vectors(N * K // v, v, "noisy", seed=3)                        # blocks of a 64 x 256 sign matrix, row-major
    C, z, info = _run(B, v, Kc, 15)
    C_ref, z_ref, _, _ = km.optimize_codebook(B, Kc, 15)
    C_pm1 = km.unpack_words(C[:info[1]], v)
    Cp = btc.codebook_pack(torch.from_numpy(np.ascontiguousarray(C_pm1)).cuda())
    idx = torch.from_numpy(z.view(np.int16).reshape(N, K // v).copy()).cuda()
    Bhat = btc.decode_pm1(idx, Cp, v, int(info[1])).cpu().numpy()
    assert (Bhat.reshape(-1, v) != B).sum() == km.total_hamming(B, C_ref, z_ref)


def test_kmeans_argument_errors():
    w = torch.zeros(16, dtype=torch.int32, device="cuda")
    with pytest.raises(btc.BtcError):
        btc.codebook_kmeans(w, 24, 16, 5)            # v > 20: unsupported
    with pytest.raises(btc.BtcError):
        btc.codebook_kmeans(w, 8, 0, 5)
    with pytest.raises(btc.BtcError):
        btc.codebook_kmeans(w, 8, 4, 0)
    with pytest.raises(btc.BtcError):
        btc.codebook_kmeans(w, 8, 4, 5, workspace=torch.empty(256, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("n,v,Kc,kind", [(30000, 20, 700, "noisy"), (200000, 16, 4096, "noisy"), (9000, 18, 3000, "iid")])
def test_kmeans_on_a_share_of_the_sms(n, v, Kc, kind):
    """On a stream of a green context of 16 SMs: a CTA per SM of the context, several parts of the patterns per CTA."""
    from cuda.bindings import driver as cu

    def ok(r):
        assert r[0] == cu.CUresult.CUDA_SUCCESS, r[0]
        return r[1:] if len(r) > 2 else r[1] if len(r) > 1 else None

    B = _vectors(n, v, kind, seed=n)
    words = torch.from_numpy(km.pack_words(B).view(np.int32).copy()).cuda()
    whole = btc.codebook_kmeans(words, v, Kc, 4)
    torch.cuda.synchronize()
    dev = ok(cu.cuDeviceGet(0))
    sm = ok(cu.cuDeviceGetDevResource(dev, cu.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(cu.cuDevSmResourceSplitByCount(1, sm, 0, 16))
    ctx = ok(cu.cuGreenCtxCreate(ok(cu.cuDevResourceGenerateDesc([groups[0]], 1)), dev, cu.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(cu.cuGreenCtxStreamCreate(ctx, cu.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    try:
        C, z, info = torch.empty_like(whole[0]), torch.empty_like(whole[1]), torch.empty_like(whole[2])
        ws = torch.empty(btc.lib.btc_codebook_kmeans_workspace_bytes(v, Kc), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        assert btc.lib.btc_codebook_kmeans(words.data_ptr(), n, v, Kc, 4, C.data_ptr(), z.data_ptr(), info.data_ptr(), ws.data_ptr(), ws.numel(), int(stream)) == 0
        torch.cuda.synchronize()
        for a, b in zip((C, z, info), whole):
            assert torch.equal(a, b)
    finally:
        torch.cuda.synchronize()
        ok(cu.cuStreamDestroy(stream))
        ok(cu.cuGreenCtxDestroy(ctx))
    assert btc.device_status() == 0
