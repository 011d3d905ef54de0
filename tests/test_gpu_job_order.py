"""Population calls with more cluster jobs than clusters fit take the longest
lattices first, a cluster per job: every candidate's actions are the bits of
its own evo_denoise call on the same decomposition."""
import numpy as np
import pytest

from paper_2607_20293_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cluster,job_samples,P,N", [(16, 1, 9, 1), (16, 2, 9, 2), (4, 1, 13, 3)])
def test_longest_first_keeps_every_candidate(cluster, job_samples, P, N):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_20293_gb300 import binding as B, build
    build.build()
    cfg = synth.config("pusht", n_steps=20, n_layer=2)
    W = synth.make_weights(cfg, 0)
    obs = torch.from_numpy(synth.make_obs(cfg, N, 5)).cuda()
    noise = torch.from_numpy(synth.make_noise(cfg, N, 6)).cuda()
    pop = np.stack([synth.bernoulli_schedule(6, 20, (p * 5 % P) / P, 30 + p) for p in range(P)])
    ev = B.Evo(cfg, W, (P + 1) * N, cluster=cluster, job_samples=job_samples, wide_rows=-1)
    x, dev = ev.population(obs, noise, pop)
    info = ev.launch_info()
    assert info["cluster"] == cluster and (P + 1) * N // job_samples > info["max_clusters"]
    x = x.cpu().numpy()
    for p in range(P):
        assert np.array_equal(x[p], ev.denoise(obs, noise, pop[p]).cpu().numpy()), p
    full = ev.denoise(obs, noise, np.ones((6, 20), np.uint8)).cpu().numpy()
    want = np.linalg.norm((x - full[None]).reshape(P, N, -1), axis=2).mean(1)
    assert np.allclose(dev.cpu().numpy(), want, rtol=1e-4, atol=1e-5)
