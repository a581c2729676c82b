"""PQ construction on the GPU vs the oracle: the encoder decides in float32
with the oracle's fixed operation order, so codes and minimum distances are
compared bit for bit; a Lloyd iteration's new centroids (fp64 means rounded
to float32, summed in another order) within one float32 ulp."""
import numpy as np
import pytest

from paper_2607_22922_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ifvs():
    from paper_2607_22922_gb300 import build
    build.build()
    from paper_2607_22922_gb300 import ifvs as mod
    return mod


def _data(w, n, seed):
    w = synth.scaled(w, N=n)
    X = synth.mixture_vectors(w, synth.mixture_centres(w))
    rng = np.random.default_rng(seed)
    C0 = X[rng.choice(n, w.K, replace=False)].reshape(w.K, w.M, w.ds).transpose(1, 0, 2).copy()
    return X, C0


CASES = [("gmm10k-d128-m16", 20_011), ("sift1m-d128-m16", 30_007), ("deep10m-d96-m12", 12_345),
         ("gist1m-d960-m120", 3_001)]


@pytest.mark.parametrize("name,n", CASES)
def test_encode_bit_exact(ifvs, orc, name, n):
    X, C0 = _data(synth.WORKLOADS[name], n, 1)
    codes, dmin = ifvs.ifvs_pq_encode(X, C0, want_dmin=True)
    rc, rd = orc.pq_encode_f32(X, C0)
    np.testing.assert_array_equal(codes, rc)
    np.testing.assert_array_equal(dmin, rd)


def test_encode_ragged_and_small_codebooks(ifvs, orc):
    rng = np.random.default_rng(4)
    for n, M, K, ds in ((1, 1, 1, 1), (33, 3, 5, 3), (257, 4, 16, 2), (1000, 2, 256, 12)):
        X = rng.standard_normal((n, M * ds)).astype(np.float32)
        C = rng.standard_normal((M, K, ds)).astype(np.float32)
        C[:, -1] = C[:, 0]                       # duplicate codeword: ties go to 0
        codes, dmin = ifvs.ifvs_pq_encode(X, C, want_dmin=True)
        rc, rd = orc.pq_encode_f32(X, C)
        np.testing.assert_array_equal(codes, rc)
        np.testing.assert_array_equal(dmin, rd)


def _hard_rows(rng, n, M, ds):
    """Rows of every scale the tensor-core ranking has a rule for: ordinary,
    far from the origin (many candidates), tiny, huge, zero, not finite."""
    X = rng.standard_normal((n, M * ds)).astype(np.float32)
    kind = rng.integers(0, 40, n)
    X[kind == 0] += 1000.0
    X[kind == 1] *= 1e-15
    X[kind == 2] *= 1e18
    X[kind == 3] = 0.0
    X[kind == 4, ::7] = np.nan
    X[kind == 5, ::5] = np.inf
    X[kind == 6] += 30.0
    return X


@pytest.mark.parametrize("ds", [4, 8, 16])
@pytest.mark.parametrize("n,M,K", [(1, 1, 1), (127, 2, 5), (128, 3, 32), (129, 5, 33), (2049, 16, 256), (300, 33, 100),
                                   (40_000, 3, 255)])
def test_encode_edges_of_the_tensor_core_path(ifvs, orc, ds, n, M, K):
    rng = np.random.default_rng(n * ds + K)
    X = _hard_rows(rng, n, M, ds)
    C = rng.standard_normal((M, K, ds)).astype(np.float32)
    C[:, -1] = C[:, 0]                           # duplicate codeword: ties go to 0
    if M > 2:
        C[1] += 500.0                            # a subspace far from the origin
        C[2, K // 2] = np.inf                    # one whose error bound does not hold
        X[:, ds:2 * ds] += 500.0
    codes, dmin = ifvs.ifvs_pq_encode(X, C, want_dmin=True)
    rc, rd = orc.pq_encode_f32(X, C)
    np.testing.assert_array_equal(codes, rc)
    np.testing.assert_array_equal(dmin, rd)
    np.testing.assert_array_equal(ifvs.ifvs_pq_encode(X, C), rc)   # without distances: fewer exact evaluations


def _hard_subspaces(rng, n, K, ds):
    """Seven subspaces: ordinary; far from the origin; very far; all zeros
    (either sign); three distinct codewords, one of them at the rows' place;
    some codewords not finite; the first codeword not finite."""
    X = rng.standard_normal((n, 7, ds), dtype=np.float32)
    C = rng.standard_normal((7, K, ds)).astype(np.float32)
    X[:, 1] += 40.0
    C[1] += 40.0
    X[:, 2] = X[:, 2] * 0.1 - 3000.0
    C[2] = C[2] * 0.1 - 3000.0
    X[:, 3] = np.copysign(0.0, X[:, 3])
    C[3] = np.copysign(0.0, C[3])
    C[4] = C[4, rng.integers(0, 3, K)]
    X[::3, 4] = C[4, K - 1]
    C[5, 3::5, ds - 1] = np.inf
    C[5, 4::9, 0] = np.nan
    C[6, 0, 1] = rng.choice([np.nan, np.inf])
    X[::1001] = np.inf
    X[5::1001, :, ds // 2] = np.nan
    return X.reshape(n, 7 * ds), C


@pytest.mark.parametrize("ds,K,n", [(4, 33, 1_250_000), (4, 256, 640_000), (8, 129, 70_001), (8, 256, 127), (16, 256, 30_001),
                                    (16, 128, 2_000)])
def test_encode_far_and_degenerate_subspaces(ifvs, orc, ds, K, n):
    """Bit for bit, several tiles per CTA and one, in the encoder's layout and
    (through a Lloyd step's objective) by subspace."""
    rng = np.random.default_rng(ds * K)
    X, C = _hard_subspaces(rng, n, K, ds)
    codes, dmin = ifvs.ifvs_pq_encode(X, C, want_dmin=True)
    rc, rd = orc.pq_encode_f32(X, C)
    np.testing.assert_array_equal(codes, rc)
    np.testing.assert_array_equal(dmin, rd)
    fin = np.isfinite(X).all(1)
    X[~fin] = 1.0                                # finite rows: finite objectives where the codebook is
    _, obj = ifvs.ifvs_pq_train(X, C, 1)
    robj = orc.pq_encode_f32(X, C)[1].astype(np.float64).sum(0)
    np.testing.assert_allclose(obj[0], robj, rtol=1e-12)


def test_encode_time_does_not_hang_on_the_data(ifvs):
    """Data that the ranking has rules for take no multiple of the time of
    ordinary data (they took six times as long when every row went through
    all codewords)."""
    import time
    import torch
    n, M, K, ds = 1 << 18, 16, 256, 8
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.randn((n, M * ds), device="cuda", generator=g)
    C = torch.randn((M, K, ds), device="cuda", generator=g)
    codes = torch.empty((n, M), dtype=torch.uint8, device="cuda")

    def ms(x, c):
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ifvs.ifvs_pq_encode(x, c, codes=codes, flags=ifvs.IFVS_F_DEVICE_IO)
            best = min(best, time.perf_counter() - t0)
        return best * 1000.0

    plain = ms(X, C)
    inf = C.clone()
    inf[:, 7, 3] = float("inf")
    for x, c in ((X + 100.0, C + 100.0), (X * 0.0, C * 0.0), (X * float("nan"), C), (X, inf),
                 (X, C[:, torch.arange(K, device="cuda") % 3].contiguous())):
        assert ms(x, c) < 2.5 * plain


def test_encode_unaligned_device_pointers(ifvs, orc):
    import torch
    rng = np.random.default_rng(9)
    n, M, K, ds = 700, 4, 64, 8
    X = rng.standard_normal((n, M * ds)).astype(np.float32)
    C = rng.standard_normal((M, K, ds)).astype(np.float32)
    x = torch.zeros(X.size + 1, device="cuda")[1:].view(n, M * ds)
    x.copy_(torch.from_numpy(X))
    c = torch.from_numpy(C).cuda()
    codes = torch.empty((n * M + 3,), dtype=torch.uint8, device="cuda")[3:].view(n, M)
    ifvs.ifvs_pq_encode(x, c, codes=codes, flags=ifvs.IFVS_F_DEVICE_IO)
    np.testing.assert_array_equal(codes.cpu().numpy(), orc.pq_encode_f32(X, C)[0])


def _ulp_close(a, b):
    a = np.asarray(a, np.float32)
    b = np.asarray(b, np.float32)
    return np.abs(a.astype(np.float64) - b.astype(np.float64)) <= np.spacing(np.maximum(np.abs(a), np.abs(b)))


@pytest.mark.parametrize("name,n", CASES[:3])
def test_one_lloyd_step(ifvs, orc, name, n):
    X, C0 = _data(synth.WORKLOADS[name], n, 2)
    C1, obj = ifvs.ifvs_pq_train(X, C0, 1)
    R1, _, robj = orc.lloyd_step(X, C0)
    assert _ulp_close(C1, R1).all()
    np.testing.assert_allclose(obj[0], robj, rtol=1e-12)


@pytest.mark.parametrize("n,M,K,ds", [(1, 3, 2, 8), (1023, 16, 256, 8), (40_003, 64, 32, 4), (9001, 2, 256, 12)])
def test_one_lloyd_step_edges(ifvs, orc, n, M, K, ds):
    """One row, one short chunk, chunks of several sorted runs, a generic
    sub-vector length; some codewords start unused."""
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, M * ds)).astype(np.float32)
    C0 = rng.standard_normal((M, K, ds)).astype(np.float32)
    C0[:, K // 2] += 50.0
    C0[:, K - 1] -= 50.0
    if n == 40_003:
        X[::7, :4] *= 1e37                       # member sums beyond float32
        X[3, 5] = np.inf
    C1, obj = ifvs.ifvs_pq_train(X, C0, 1)
    R1, _, robj = orc.lloyd_step(X, C0)
    with np.errstate(invalid="ignore"):
        assert (_ulp_close(C1, R1) | (C1 == R1) | (np.isnan(C1) & np.isnan(R1))).all()
    np.testing.assert_allclose(obj[0], robj, rtol=1e-12)


def test_lloyd_sums_of_long_lopsided_runs(ifvs, orc):
    """Runs of half a million members per chunk whose rounding errors do not
    cancel (a constant, nearly one value, one sign): the float64 means to one
    ulp, and the objective (errors of 10^6 additions of one sign, sqrt(n)
    2^-53 to n 2^-53 = 1e-13 to 1e-10, exact for the alike values)."""
    rng = np.random.default_rng(12)
    n, M = 1_000_000, 120
    X = rng.standard_normal((n, M), dtype=np.float32)
    X[:, 0] = 0.1
    X[:, 1] = 0.3
    X[:, 2] = 0.3 + 1e-4 * X[:, 2]
    X[:, 3] = 1.7 + 0.025 * rng.random(n, dtype=np.float32)
    X[:, 4] = np.abs(X[:, 4])
    X[:, 5] = np.exp(2.0 * X[:, 5])
    C0 = np.zeros((M, 2, 1), np.float32)
    C0[:, 0] = 0.45
    C0[:, 1] = 2000.0                            # takes nothing, or the tail of the lognormal
    C1, obj = ifvs.ifvs_pq_train(X, C0, 1)
    R1, codes, robj = orc.lloyd_step(X, C0)
    assert (codes[:, :5] == 0).all()
    assert _ulp_close(C1, R1).all(), np.argwhere(~_ulp_close(C1, R1))
    np.testing.assert_allclose(obj[0, :4], robj[:4], rtol=1e-12)
    np.testing.assert_allclose(obj[0], robj, rtol=1e-10)


def _step_ms(ifvs, X, C, iters=2):
    """Fastest of three calls of `iters` Lloyd steps on device data, in ms per step."""
    import time
    import torch
    out = torch.empty_like(C)
    best = 1e9
    for _ in range(4):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ifvs.ifvs_pq_train(X, C, iters, C_out=out, flags=ifvs.IFVS_F_DEVICE_IO)
        best = min(best, time.perf_counter() - t0)
    return best * 1000.0 / iters


def test_a_lloyd_step_is_not_slowed_down_by_an_infinite_value(ifvs, orc):
    """One infinite value per sub-vector of 2^20 rows: the sums that hold it are
    infinite, the others right, and the step takes no multiple of its time
    (a thread that went over all rows again took 17 times as long)."""
    import torch
    rng = np.random.default_rng(4)
    n, M, K, ds = 1 << 20, 4, 256, 8
    X = rng.standard_normal((n, M * ds), dtype=np.float32)
    C = np.ascontiguousarray(X[:K].reshape(K, M, ds).transpose(1, 0, 2))
    plain = _step_ms(ifvs, torch.from_numpy(X).cuda(), torch.from_numpy(C).cuda())
    X[1234, ::ds] = np.inf
    assert _step_ms(ifvs, torch.from_numpy(X).cuda(), torch.from_numpy(C).cuda()) < 4.0 * plain
    G, obj = ifvs.ifvs_pq_train(X, C, 1)
    R, _, robj = orc.lloyd_step(X, C)
    with np.errstate(invalid="ignore"):
        assert (_ulp_close(G, R) | (G == R) | (np.isnan(G) & np.isnan(R))).all()
    assert np.isinf(G).any() and np.isinf(obj).all() and np.isinf(robj).all()


def test_a_lloyd_step_of_more_subspaces_than_a_grid_dimension_has(ifvs, orc):
    import torch
    rng = np.random.default_rng(6)
    M = 66_000
    X = rng.standard_normal((40, M)).astype(np.float32)
    C = rng.standard_normal((M, 2, 1)).astype(np.float32)
    out = torch.empty((M, 2, 1), device="cuda")
    ifvs.ifvs_pq_train(torch.from_numpy(X).cuda(), torch.from_numpy(C).cuda(), 1, C_out=out, flags=ifvs.IFVS_F_DEVICE_IO)
    R, _, _ = orc.lloyd_step(X, C)
    assert _ulp_close(out.cpu().numpy(), R).all()


def test_empty_codewords_take_the_farthest_points(ifvs, orc):
    rng = np.random.default_rng(5)
    X = rng.standard_normal((4000, 16)).astype(np.float32)
    C0 = rng.standard_normal((2, 64, 8)).astype(np.float32)
    C0[:, 40:] += 100.0                          # 24 codewords per subspace attract nobody
    C1, _ = ifvs.ifvs_pq_train(X, C0, 1)
    R1, codes, _ = orc.lloyd_step(X, C0)
    assert (np.bincount(codes[:, 0], minlength=64)[40:] == 0).all()
    assert _ulp_close(C1, R1).all()


def test_lloyd_iterations_track_the_oracle(ifvs, orc):
    X, C = _data(synth.WORKLOADS["gmm10k-d128-m16"], 8_000, 3)
    G, gobj = ifvs.ifvs_pq_train(X, C, 5)
    R = C
    for it in range(5):
        R, _, robj = orc.lloyd_step(X, R)
        np.testing.assert_allclose(gobj[it], robj, rtol=1e-9)
    assert (np.diff(gobj, axis=0) <= 1e-6 * gobj[:-1]).all()
    assert _ulp_close(G, R).mean() > 0.999


def test_device_io_on_a_caller_stream(ifvs, orc):
    import torch
    X, C0 = _data(synth.WORKLOADS["gmm10k-d128-m16"], 9_999, 6)
    dev = torch.device("cuda", 0)
    s = torch.cuda.Stream(device=dev)
    Xd, Cd = torch.from_numpy(X).to(dev), torch.from_numpy(C0).to(dev)
    codes = torch.empty((len(X), C0.shape[0]), dtype=torch.uint8, device=dev)
    dmin = torch.empty((len(X), C0.shape[0]), dtype=torch.float32, device=dev)
    torch.cuda.synchronize()
    ifvs.ifvs_pq_encode(Xd, Cd, codes=codes, dmin=dmin, flags=ifvs.IFVS_F_DEVICE_IO,
                        stream=s.cuda_stream)
    s.synchronize()
    rc, rd = orc.pq_encode_f32(X, C0)
    np.testing.assert_array_equal(codes.cpu().numpy(), rc)
    np.testing.assert_array_equal(dmin.cpu().numpy(), rd)
    C1 = torch.empty_like(Cd)
    obj = torch.empty((2, C0.shape[0]), dtype=torch.float64, device=dev)
    ifvs.ifvs_pq_train(Xd, Cd, 2, C_out=C1, objective=obj, flags=ifvs.IFVS_F_DEVICE_IO,
                       stream=s.cuda_stream)
    H1, hobj = ifvs.ifvs_pq_train(X, C0, 2)
    np.testing.assert_array_equal(C1.cpu().numpy(), H1)
    np.testing.assert_array_equal(obj.cpu().numpy(), hobj)


def test_device_io_without_a_stream_orders_after_default_stream_work(ifvs):
    """With device I/O and no stream, the call runs on a stream of the
    library's own that must wait for the caller's pending work on the legacy
    default stream: vectors computed there by torch right before the call
    (no synchronisation in between) are encoded as if the call had waited."""
    import torch
    dev = torch.device("cuda", 0)
    torch.cuda.synchronize()
    M, K, ds, n = 16, 256, 8, 1 << 21
    with torch.cuda.stream(torch.cuda.default_stream(dev)):
        g = torch.Generator(device=dev)
        g.manual_seed(11)
        C = torch.randn((M, K, ds), generator=g, device=dev)
        for rep in range(3):
            torch.cuda.synchronize()
            # long default-stream work that produces X, then the call at once
            X = torch.randn((n, M * ds), generator=g, device=dev)
            for _ in range(4):
                X = torch.tanh(X * 1.5) * 2.0
            codes = torch.empty((n, M), dtype=torch.uint8, device=dev)
            ifvs.ifvs_pq_encode(X, C, codes=codes, flags=ifvs.IFVS_F_DEVICE_IO, stream=None)
            torch.cuda.synchronize()
            again = torch.empty_like(codes)
            ifvs.ifvs_pq_encode(X, C, codes=again, flags=ifvs.IFVS_F_DEVICE_IO, stream=None)
            torch.cuda.synchronize()
            assert torch.equal(codes, again), "the encode read X before it was written (rep %d)" % rep
