"""GPU parity of the redundancy-aware initialisation: the dissimilarity map of
Eq. 6 and its variants (evo_redundancy_map) and guided sampling (Eq. 7,
evo_guided_schedules) against the float64 oracle.

The map is compared on the same activations (the oracle's all-refresh trace,
and synthetic activations for the larger shapes) to 1e-5 absolute plus 1e-4
relative (fp32 sums of n products), and end to end from the GPU's own trace;
the schedules must be identical bit for bit (integer arithmetic)."""
import numpy as np
import pytest

from oracle import evo_oracle as O
from paper_2607_20293_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    return _t


@pytest.fixture(scope="module")
def B(torch):
    from paper_2607_20293_gb300 import binding, build
    build.build()
    binding.load()
    return binding


@pytest.fixture(scope="module")
def tiny_trace():
    cfg = synth.config("tiny")
    W = synth.make_weights(cfg, 0)
    n = 3
    obs, noise = synth.make_obs(cfg, n, 11), synth.make_noise(cfg, n, 12)
    U, T = 3 * cfg["n_layer"], cfg["n_steps"]
    tr = {}
    O.denoise(W, cfg, obs, noise, np.ones((U, T), np.uint8), trace=tr)
    return cfg, W, obs, noise, O.trace_activations(tr, U, T)


def _close(got, want):
    got = np.asarray(got, np.float64)
    assert np.all(np.isfinite(got))
    assert np.allclose(got, want, atol=1e-5, rtol=1e-4), float(np.max(np.abs(got - want)))


@pytest.mark.parametrize("metric", ["cosine", "mse", "l1", "w1"])
def test_map_on_oracle_trace(torch, B, tiny_trace, metric):
    cfg, W, obs, noise, acts = tiny_trace
    trace = np.ascontiguousarray(acts.transpose(2, 1, 0, 3, 4), dtype=np.float32)   # [T][U][N][H][E]
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), metric).cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3, 4).astype(np.float64), metric))


def test_map_end_to_end_from_gpu_trace(torch, B, tiny_trace):
    cfg, W, obs, noise, acts = tiny_trace
    U, T, H, E = 3 * cfg["n_layer"], cfg["n_steps"], cfg["horizon"], cfg["n_emb"]
    ev = B.Evo(cfg, W, 3)
    tr = torch.zeros((T, U, 3, H, E), device="cuda")
    ev.denoise(torch.from_numpy(obs).cuda(), torch.from_numpy(noise).cuda(), np.ones((U, T), np.uint8), trace=tr)
    got = B.redundancy_map(tr, "cosine").cpu().numpy()
    _close(got, O.redundancy_map(acts, "cosine"))


@pytest.mark.parametrize("metric", ["cosine", "w1"])
def test_map_push_t_sized_rows(torch, B, metric):
    # n = 16 x 256 entries per activation (Push-T-shaped), several chunks of the pair kernel
    rng = np.random.default_rng(21)
    T, U, N, n = 20, 4, 2, 4096
    base = rng.standard_normal((U, N, n))
    trace = (base[None] + 0.3 * rng.standard_normal((T, U, N, n))).astype(np.float32)
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), metric).cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3).astype(np.float64), metric))


@pytest.mark.parametrize("metric", ["mse", "l1"])
def test_map_ragged_rows(torch, B, metric):
    # n = 77 entries: a partial chunk and rows that are not 16-byte multiples
    rng = np.random.default_rng(22)
    T, U, N, n = 7, 3, 2, 77
    trace = rng.standard_normal((T, U, N, n)).astype(np.float32)
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), metric).cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3).astype(np.float64), metric))


def test_map_rejects_bad_shapes(torch, B):
    assert B.load().evo_redundancy_scratch_bytes(1, 4, 2, 64, 0) == 0          # T < 2
    assert B.load().evo_redundancy_scratch_bytes(10, 4, 2, 100, 3) == 0        # w1 needs a power of two
    assert B.load().evo_redundancy_scratch_bytes(10, 4, 2, 100, 0) > 0


@pytest.mark.parametrize("K,eps,gamma", [(120, 0.05, 2), (0, 0.05, 2), (800, 0.05, 2), (37, 0.0, 1), (300, 0.2, 3)])
def test_guided_schedules_bit_exact(torch, B, K, eps, gamma):
    d = synth.dissimilarity_map(8, 100, 5).astype(np.float32)
    P = 16
    rnd = synth.guided_randoms(P, max(K, 1), 7)
    got = B.guided_schedules(torch.from_numpy(d).cuda(), K, torch.from_numpy(rnd.view(np.int64)).cuda(),
                             eps, gamma).cpu().numpy()
    want = O.guided_schedules(d, K, eps, gamma, rnd)
    assert np.array_equal(got, want)
    assert np.all(got.reshape(P, -1).sum(1) == K)


def test_guided_schedules_zero_weights(torch, B):
    # eps = 0 with zero map entries: zero weights are drawn only when nothing else is left
    d = np.zeros((4, 10), np.float32)
    d[1, 3], d[2, 7] = 1.0, 0.5
    rnd = synth.guided_randoms(4, 5, 8)
    got = B.guided_schedules(torch.from_numpy(d).cuda(), 5, torch.from_numpy(rnd.view(np.int64)).cuda(), 0.0,
                             1).cpu().numpy()
    assert np.array_equal(got, O.guided_schedules(d, 5, 0.0, 1, rnd))
    assert np.all(got[:, 1, 3] == 1) and np.all(got[:, 2, 7] == 1)


@pytest.mark.parametrize("units,steps,K", [(1, 1, 1), (3, 10, 30), (1, 33, 7), (5, 51, 255), (24, 100, 240), (32, 128, 500)])
def test_guided_schedules_run_edges(torch, B, units, steps, K):
    # fewer cells than lanes, runs that do not divide the cells, every cell drawn, the largest lattice
    rng = np.random.default_rng(units * steps)
    d = (rng.random((units, steps)) + 0.01).astype(np.float32)
    rnd = synth.guided_randoms(3, K, 9)
    got = B.guided_schedules(torch.from_numpy(d).cuda(), K, torch.from_numpy(rnd.view(np.int64)).cuda(), 0.05,
                             2).cpu().numpy()
    assert np.array_equal(got, O.guided_schedules(d, K, 0.05, 2, rnd))


def _wrapping_draws(q, K, rnd):
    """Draws on 64-bit sums that wrap: the first of 32 runs of cells whose last running
    sum exceeds the target, in it the first cell whose running sum does."""
    M = 1 << 64
    ch = (len(q) + 31) // 32
    left = [int(v) for v in q]
    out = np.zeros(len(q), np.uint8)
    for k in range(K):
        run, sums = 0, []
        for v in left:
            run = (run + v) % M
            sums.append(run)
        target = int(rnd[k]) % sums[-1]
        lo = next(i for i in range(0, len(q), ch) if sums[min(i + ch, len(q)) - 1] > target)
        pick = next(i for i in range(lo, lo + ch) if sums[i] > target)
        out[pick], left[pick] = 1, 0
    return out


@pytest.mark.parametrize("eps,gamma", [(10.0, 4), (30.0, 4), (45.0, 4), (7.0, 7)])
def test_guided_schedules_wrapping_sums(torch, B, eps, gamma):
    # 2,400 weights whose sum passes 2^64, in the last three the sum of every run of 75 cells too
    d = synth.dissimilarity_map(24, 100, 5).astype(np.float32)
    q = O.guided_weights(d, eps, gamma)
    assert sum(int(v) for v in q) > 1 << 64
    P, K = 8, 60
    rnd = synth.guided_randoms(P, K, 17)
    got = B.guided_schedules(torch.from_numpy(d).cuda(), K, torch.from_numpy(rnd.view(np.int64)).cuda(), eps,
                             gamma).cpu().numpy()
    want = np.stack([_wrapping_draws(q, K, rnd[p]).reshape(d.shape) for p in range(P)])
    assert np.array_equal(got, want)


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384])
def test_map_w1_row_lengths(torch, B, n):
    # every register-sort size (several rows per block and one) and the shared-memory sort below them;
    # a last block with idle rows
    rng = np.random.default_rng(n)
    T, U, N = 4, 3, 1
    trace = rng.standard_normal((T, U, N, n)).astype(np.float32)
    trace[1, 0, 0, : n // 2] = 0.0                                  # ties
    trace[2, 1, 0] = -np.abs(trace[2, 1, 0])
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), "w1").cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3).astype(np.float64), "w1"))


def test_map_w1_keeps_nan_and_inf(torch, B):
    # a sort that lost a NaN would give its row, and every row's mean, finite values
    rng = np.random.default_rng(3)
    trace = rng.standard_normal((4, 3, 1, 256)).astype(np.float32)
    trace[2, 0, 0, 17] = np.nan
    trace[1, 1, 0, 200] = np.inf
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), "w1").cpu().numpy()
    assert np.all(np.isnan(got[0])) and np.all(np.isinf(got[1])) and np.all(np.isfinite(got[2]))


def _entry_order_l1(trace):
    """The mean-absolute-difference map in fp32, every sum in index order:
    a pair's over the entries, a row's over the steps, the mean over the samples."""
    T, U, N, n = trace.shape
    d = np.zeros((U, T), np.float32)
    for r in range(N):
        x = trace[:, :, r]                                          # [T][U][n]
        g = np.zeros((T, T, U), np.float32)
        for k in range(n):
            g += np.abs(x[:, None, :, k] - x[None, :, :, k])
        g /= np.float32(n)
        s = np.zeros((T, U), np.float32)
        for t2 in range(T):
            s += np.where(np.arange(T)[:, None] == t2, np.float32(0), g[:, t2])
        d += (s / np.float32(T - 1)).T
    return d / np.float32(N)


@pytest.mark.parametrize("T,n", [(2, 64), (8, 256), (32, 128), (33, 256), (64, 512), (65, 256), (100, 1024), (128, 256)])
def test_map_w1_bits_in_entry_order(torch, B, T, n):
    # a map that differs in its last bits draws other guided schedules: the sorted
    # rows' sums run in entry order in every tile shape, and a unit's map does not
    # depend on which units share the call
    rng = np.random.default_rng(T + n)
    trace = rng.standard_normal((T, 4, 2, n)).astype(np.float32)
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), "w1").cpu().numpy()
    assert np.array_equal(got, _entry_order_l1(np.sort(trace, axis=-1)))
    one = B.redundancy_map(torch.from_numpy(np.ascontiguousarray(trace[:, 1:2])).cuda(), "w1").cpu().numpy()
    assert np.array_equal(one[0], got[1])


@pytest.mark.parametrize("metric", ["cosine", "mse", "l1", "w1"])
@pytest.mark.parametrize("T,n", [(2, 3), (7, 64), (8, 256), (9, 260), (32, 516), (33, 130), (64, 64), (65, 77), (100, 1028),
                                 (128, 333)])
def test_map_tile_edges(torch, B, metric, T, n):
    # the three tile shapes and the step counts where they change (32 | 33, 64 | 65), row
    # groups of four filled in part, one chunk of 32 entries and several, a ragged last one
    if metric == "w1":
        n = 1 << (n - 1).bit_length()                               # the sorted rows' lengths
    rng = np.random.default_rng(T * 1000 + n)
    U, N = 2, 2
    base = rng.standard_normal((U, N, n))
    trace = (base[None] + 0.5 * rng.standard_normal((T, U, N, n))).astype(np.float32)
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), metric).cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3).astype(np.float64), metric))


def test_map_w1_odd_number_of_maps(torch, B):
    # 7 x 3 x 1 per-sample values in front of the sorted rows
    rng = np.random.default_rng(5)
    trace = rng.standard_normal((7, 3, 1, 512)).astype(np.float32)
    got = B.redundancy_map(torch.from_numpy(trace).cuda(), "w1").cpu().numpy()
    _close(got, O.redundancy_map(trace.transpose(2, 1, 0, 3).astype(np.float64), "w1"))


@pytest.mark.parametrize("metric", ["cosine", "mse", "l1", "w1"])
def test_map_rows_off_16_bytes(torch, B, metric):
    # a trace and a scratch of the caller's that start 4 bytes off: the rows are read by plain loads
    rng = np.random.default_rng(6)
    T, U, N, n = 40, 3, 1, 256
    trace = rng.standard_normal((T, U, N, n)).astype(np.float32)
    m = B.METRICS[metric]
    nb = B.load().evo_redundancy_scratch_bytes(T, U, N, n, m)
    buf = torch.empty(trace.size + 1, device="cuda")
    buf[1:] = torch.from_numpy(trace).cuda().flatten()
    scratch = torch.empty(nb // 4 + 1, device="cuda")
    d = torch.empty((U, T), device="cuda")
    assert B.load().evo_redundancy_map(buf[1:].data_ptr(), T, U, N, n, m, d.data_ptr(), scratch[1:].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream) == B.OK
    want = B.redundancy_map(torch.from_numpy(trace).cuda(), metric)
    assert torch.equal(d, want)
