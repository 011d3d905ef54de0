"""GPU parity of the tile path (one block runs the whole loop of up to 8 samples)
against the float64 oracle: the library's own choice from 128 samples (2,048
action-token rows) on for n_emb 256, horizon 16.

Cases are the edges of its tiles and operands: a last tile of 1 .. 8 samples,
1 and 16 actions, 1 and 7 observation tokens (2 and 8 memory keys), both
samplers and empty-cache policies, coarse and device lattices, lattices that
refresh nothing, one cell or everything.  Tolerance: max-abs 3e-2 on final
actions (bf16 mode), on sampled chunks."""
import numpy as np
import pytest

from eq1_trace import check_reuse
from oracle import evo_oracle as O
from paper_2607_20293_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 3e-2


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


def on_tiles(ev):
    info = ev.launch_info()
    return info["cluster"] == 1 and info["job_samples"] == 8


def close(got, want, what=""):
    assert np.all(np.isfinite(got)), what
    err = float(np.max(np.abs(got - want)))
    assert err <= TOL, f"{what}: max-abs {err:.3e}"


# 128 = 16 full tiles, 129 = a last tile of one sample, 506 = of 2, 133 = of 5, 231 = of 7
@pytest.mark.parametrize("n,over,frac", [
    (133, {}, 0.3),
    (128, dict(action_dim=16, n_obs=7, obs_dim=30), 1.0),
    (129, dict(action_dim=1, n_obs=1), 0.3),
    (231, dict(sampler="ddim", n_layer=1), 0.5),
    (506, dict(n_layer=2, action_dim=5), 0.05),
])
def test_tile_matches_oracle(torch, B, n, over, frac):
    cfg = synth.config("pusht", n_steps=20, **over)
    units = 3 * cfg["n_layer"]
    W = synth.make_weights(cfg, 0)
    obs, noise = synth.make_obs(cfg, n, 71), synth.make_noise(cfg, n, 72)
    S = np.ones((units, 20), np.uint8) if frac == 1.0 else synth.bernoulli_schedule(units, 20, frac, 73)
    ev = B.Evo(cfg, W, n)
    got = ev.denoise(torch.from_numpy(obs).cuda(), torch.from_numpy(noise).cuda(), S).cpu().numpy()
    assert on_tiles(ev)
    # the blocks that are resident at once, one per SM, however many tiles the call has
    assert ev.launch_info()["max_clusters"] == torch.cuda.get_device_properties(0).multi_processor_count
    idx = [0, 7, 8, n - 2, n - 1]
    close(got[idx], O.denoise(W, cfg, obs[idx], noise[:, idx], S), f"n={n}")
    assert ev.status() == B.OK


@pytest.mark.parametrize("empty", ["zero", "force"])
def test_tile_population_edge_lattices(torch, B, empty):
    # 11 observations: a tile of 8 samples and one of 3 per lattice
    cfg = synth.config("pusht", n_steps=20, n_layer=2)
    U, T, N = 6, 20, 11
    W = synth.make_weights(cfg, 0)
    P = 40
    lat = np.zeros((P, U, T), np.uint8)
    lat[0, 0, 0] = 1                  # the first cell only
    lat[1, U - 1, T - 1] = 1          # the last cell only
    lat[2, :, 0] = 1                  # every unit at step 0, then skips to the end
    lat[3, :, T - 1] = 1
    lat[4] = 1                        # the reference itself; lattice 5: nothing refreshed
    for p in range(6, P):
        lat[p] = synth.bernoulli_schedule(U, T, 0.1 * (p % 11), p)
    obs, noise = synth.make_obs(cfg, N, 81), synth.make_noise(cfg, N, 82)
    ev = B.Evo(cfg, W, (P + 1) * N, empty=empty)
    x, dev = ev.population(torch.from_numpy(obs).cuda(), torch.from_numpy(noise).cuda(), lat)
    assert on_tiles(ev)
    x, dev = x.cpu().numpy(), dev.cpu().numpy()
    idx = [0, 7, 8, 10]
    for p in range(11):
        close(x[p][idx], O.denoise(W, cfg, obs[idx], noise[:, idx], lat[p], policy=empty), f"lattice {p} ({empty})")
    assert dev[4] == 0.0              # the same jobs on the same kernel
    full = x[4]
    want = np.linalg.norm((x - full[None]).reshape(P, N, -1), axis=2).mean(1)
    assert np.allclose(dev, want, rtol=1e-4, atol=1e-5)
    # a few short lattices stay on tiles (132 samples), which keep the partial sums that cross
    # a cluster in bf16 in fp32, with the same bits wherever the lattices live
    for lattices in (lat[:11], torch.from_numpy(lat[:11]).cuda()):
        x2, _ = ev.population(torch.from_numpy(obs).cuda(), torch.from_numpy(noise).cuda(), lattices)
        assert on_tiles(ev)
        assert np.array_equal(x2.cpu().numpy(), x[:11])


def test_tile_lattice_forms(torch, B):
    # coarse [L][T] and device lattices give the bits of the unit lattice on the
    # host; an invalid lattice is refused before anything is launched
    cfg = synth.config("pusht", n_steps=20, n_layer=2)
    n = 130
    W = synth.make_weights(cfg, 0)
    obs = torch.from_numpy(synth.make_obs(cfg, n, 91)).cuda()
    noise = torch.from_numpy(synth.make_noise(cfg, n, 92)).cuda()
    S = synth.bernoulli_schedule(2, 20, 0.7, 93)
    ev = B.Evo(cfg, W, n)
    want = ev.denoise(obs, noise, np.repeat(S, 3, axis=0)).cpu().numpy()
    assert on_tiles(ev)
    assert np.array_equal(ev.denoise(obs, noise, S).cpu().numpy(), want)
    assert np.array_equal(ev.denoise(obs, noise, torch.from_numpy(S).cuda()).cpu().numpy(), want)
    bad = torch.from_numpy(S).cuda()
    bad[1, 3] = 2
    out = torch.full((n, 16, 2), 5.0, device="cuda")
    for lattice in (bad, bad.cpu().numpy()):
        with pytest.raises(B.EvoError) as e:
            ev.denoise(obs, noise, lattice, out=out)
        assert e.value.code == B.ERR_SCHEDULE
    assert torch.all(out == 5.0) and ev.status() == B.OK


# 2 layers: the line lies at 2.8 refreshed cells a step for 128 samples, at 1.15 for 239,
# 0.4 from 240 to 499 and 0 from 500 on
@pytest.mark.parametrize("n,cells,tiles", [(128, 27, False), (128, 29, True), (239, 11, False), (239, 12, True),
                                           (240, 3, False), (240, 4, True), (499, 3, False), (500, 0, True)])
def test_one_sparse_lattice_runs_batch_wide(torch, B, n, cells, tiles):
    cfg = synth.config("pusht", n_steps=10, n_layer=2)
    W = synth.make_weights(cfg, 0)
    S = np.zeros((60,), np.uint8)
    S[np.random.default_rng(n).choice(60, cells, replace=False)] = 1
    S = S.reshape(6, 10)
    obs, noise = synth.make_obs(cfg, n, 74), synth.make_noise(cfg, n, 75)
    d_obs, d_noise = torch.from_numpy(obs).cuda(), torch.from_numpy(noise).cuda()
    ev = B.Evo(cfg, W, n)
    got = ev.denoise(d_obs, d_noise, S)
    assert ev.last_call()["path"] == ("cluster" if tiles else "wide")
    assert torch.equal(ev.denoise(d_obs, d_noise, torch.from_numpy(S).cuda()), got)
    assert ev.last_call()["path"] == ("cluster" if tiles else "wide")
    idx = [0, n - 1]
    close(got.cpu().numpy()[idx], O.denoise(W, cfg, obs[idx], noise[:, idx], S), f"n={n} cells={cells}")
    if cells % 3 == 0:                         # the same cells as rows of layers
        L = np.zeros((2, 10), np.uint8)
        L.reshape(-1)[:cells // 3] = 1
        ev.denoise(d_obs, d_noise, L)
        assert ev.last_call()["path"] == ("cluster" if tiles else "wide")


@pytest.mark.parametrize("empty", ["zero", "force"])
def test_tile_trace_takes_the_tile_path(torch, B, empty):
    # the traced call runs where the untraced one does and gives its actions bit for bit; a cell that
    # is skipped adds the stored bf16 value (Eq. 1), one that is refreshed its own output
    cfg = synth.config("pusht", n_steps=10, n_layer=2)
    n, U, T = 243, 6, 10                       # a last tile of 3 samples
    W = synth.make_weights(cfg, 0)
    S = synth.bernoulli_schedule(U, T, 0.5, 97)
    S[2] = 0                                   # a unit that is never refreshed
    S[4, :3], S[4, 3] = 0, 1                   # one whose cache stays empty at first
    obs_h, noise_h = synth.make_obs(cfg, n, 98), synth.make_noise(cfg, n, 99)
    obs, noise = torch.from_numpy(obs_h).cuda(), torch.from_numpy(noise_h).cuda()
    ev = B.Evo(cfg, W, n, empty=empty)
    want = ev.denoise(obs, noise, S)
    assert on_tiles(ev)
    tr = torch.full((T, U, n, 16, 256), float("nan"), device="cuda")
    got = ev.denoise(obs, noise, S, trace=tr)
    assert on_tiles(ev) and torch.equal(got, want) and ev.status() == B.OK
    tr = tr.cpu().numpy()
    assert np.all(np.isfinite(tr))
    assert check_reuse(tr, S, bf16=True, force=empty == "force") > 0
    idx, ref = [0, 8, n - 1], {}
    O.denoise(W, cfg, obs_h[idx], noise_h[:, idx], S, policy=empty, trace=ref)
    # (3 % of the largest: the bound on final actions, relative)
    top = max(np.max(np.abs(v)) for _, v in ref.values() if v is not None)
    for (b, t), (_, v) in ref.items():
        assert np.max(np.abs(tr[t, b][idx] - (0.0 if v is None else v))) <= TOL * top, (b, t)


def test_handles_too_small_for_tiles_hold_nothing_of_them(torch, B):
    # a handle whose largest call stays below the threshold takes no more device
    # memory than one whose threshold is fixed, which never has a tile path (its
    # packed weights alone are 14.7 MB at 8 layers)
    cfg = synth.config("pusht")
    W = synth.make_weights(cfg, 0)

    def held(n, **kw):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ev = B.Evo(cfg, W, n, **kw)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        ev.close()
        return used

    held(128), held(127, wide_rows=2048)       # the kernels' modules are loaded
    assert held(127) == held(127, wide_rows=2048)
    assert held(128) > held(128, wide_rows=2048) + 14_000_000


@pytest.mark.parametrize("n", [109, 127])
def test_calls_below_the_tile_threshold_stay_on_clusters(torch, B, n):
    # the cluster path's condition kernels and head keep their operands in fp32:
    # a handle with default options gives the bits of one that has no other path,
    # for a query batch and for a population, wherever the lattices are
    cfg = synth.config("pusht", n_steps=20, n_layer=2)
    W = {k: (v * np.float32(1.001)).astype(np.float32) for k, v in synth.make_weights(cfg, 0).items()}   # not in bf16
    obs = torch.from_numpy(synth.make_obs(cfg, n, 94)).cuda()
    noise = torch.from_numpy(synth.make_noise(cfg, n, 95)).cuda()
    S = synth.bernoulli_schedule(6, 20, 0.3, 96)
    ev, cl = B.Evo(cfg, W, n), B.Evo(cfg, W, n, wide_rows=-1)
    want = cl.denoise(obs, noise, S)
    for lattice in (S, torch.from_numpy(S).cuda()):
        assert torch.equal(ev.denoise(obs, noise, lattice), want)
        assert ev.last_call()["path"] == "cluster" and not on_tiles(ev)
    P = n - 1
    pop = np.stack([synth.bernoulli_schedule(6, 20, 0.5, 200 + p) for p in range(P)])
    o1, z1 = obs[:1].contiguous(), noise[:, :1].contiguous()
    want, want_dev = cl.population(o1, z1, pop)
    for lattice in (pop, torch.from_numpy(pop).cuda()):
        x, dev = ev.population(o1, z1, lattice)
        assert torch.equal(x, want) and torch.equal(dev, want_dev)
        assert ev.last_call()["path"] == "cluster" and not on_tiles(ev)
