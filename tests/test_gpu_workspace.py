"""The stateless calls' workspace: one pool per device that serves every stream
and thread, is made by whichever call comes first (also one that a stream
capture records), and gives its memory back when asked or needed."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from tests.gpu_util import dev, egarch_truth, host, particles, soa, torch_cuda
from paper_1304_4334_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def S():
    torch_cuda()
    from paper_1304_4334_gb300 import smc
    return smc


CAPTURE = """
import torch
from tests.gpu_util import dev, egarch_truth, particles, soa
from paper_1304_4334_gb300 import inputs as I, smc as S
K, I_, T, P = 2, 2, 50, 333
truth = egarch_truth(K, I_)
y, m = dev(I.simulate_egarch(truth, T, seed=71)), S.model_egarch(K, I_, True)
d = 2 + 3 * K + 3 * I_
clouds = [soa(particles(d, truth, K, I_, True, P, s)) for s in (1, 2)]
theta = clouds[0].clone()
def out(): return [torch.zeros(P, dtype=torch.float64, device="cuda"), torch.zeros((d, P), dtype=torch.float64, device="cuda")]
got, want = out(), out()
s = torch.cuda.Stream()
s.wait_stream(torch.cuda.current_stream())
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=s):      # the process's first stateless call
    S.loglik_grad(m, S.FP64, y, theta, *got)
for c in clouds:
    theta.copy_(c)
    g.replay()
    S.loglik_grad(m, S.FP64, y, c, *want)
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and bool(torch.isfinite(got[1]).all())
print("captured ok")
"""


def test_first_call_recorded_by_a_capture():
    torch_cuda()
    r = subprocess.run([sys.executable, "-c", CAPTURE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured ok" in r.stdout, r.stdout + r.stderr


def _work(S, torch, seed):
    """A round of calls whose workspaces differ in size, on the thread's current
    stream; returns their results."""
    rng = np.random.default_rng(seed)
    K, I_, T = 2, 2, 40
    truth = egarch_truth(K, I_)
    y, m = dev(I.simulate_egarch(truth, T, seed=71)), S.model_egarch(K, I_, True)
    d = 2 + 3 * K + 3 * I_
    out = []
    for P in (200, 30000, 3000):
        x = soa(particles(d, truth, K, I_, True, P, seed))
        ll, lp, g = (torch.zeros(n, dtype=torch.float64, device="cuda") for n in (P, P, (d, P)))
        st = torch.zeros((K + 1, P), dtype=torch.float64, device="cuda")
        mean, cov, L = (torch.zeros(n, dtype=torch.float64, device="cuda") for n in ((d,), (d, d), (d, d)))
        logw = dev(rng.normal(size=P))
        idx = torch.zeros(P, dtype=torch.int32, device="cuda")
        S.loglik(m, S.FP64, y, x, ll, lp, st)
        S.loglik_grad(m, S.FP64, y, x, ll, g, st)
        S.cov_chol(x, 3, mean, cov, L)
        n = S.mutate_rw(m, S.FP64, y, x, ll, lp, st, L, 0.3, 9, 2, 3)
        dphi, rss = S.power_search(ll, 0.3)
        lwbar = S.resample_logw(logw, 1 if P <= 4096 else 8, P if P <= 4096 else P // 8, idx, seed=3, cycle=1)
        out += [n, dphi, rss, lwbar.copy()] + [t for t in (x, ll, lp, st, g, cov, L, idx)]
    return out


def _same(torch, a, b):
    # (the RSS is NaN above the largest group)
    return all(torch.equal(u, v) if isinstance(u, torch.Tensor) else np.array_equal(u, v, equal_nan=True)
               for u, v in zip(a, b))


def test_threads_and_streams_share_the_pool(S):
    """Four threads, each on its own stream, against the same calls in a row."""
    torch = torch_cuda()
    seeds = [11, 12, 13, 14]
    want = [_work(S, torch, s) for s in seeds]
    torch.cuda.synchronize()
    got, errors = {}, []

    def run(s):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    got[s] = _work(S, torch, s)
                torch.cuda.current_stream().synchronize()
        except Exception as e:   # (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=(s,)) for s in seeds]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for s, w in zip(seeds, want):
        assert _same(torch, got[s], w), s


def test_release_workspace_gives_the_memory_back(S):
    torch = torch_cuda()
    want = _work(S, torch, 21)
    K, P, T = 2, 100000, 600          # checkpoints: 37 x 3 x P x 8 bytes = 89 MB
    truth = egarch_truth(K, 2)
    y, m = dev(I.simulate_egarch(truth, T, seed=71)), S.model_egarch(K, 2, True)
    x = soa(particles(14, truth, K, 2, True, P, 5))
    ll, g = torch.zeros(P, dtype=torch.float64, device="cuda"), torch.zeros((14, P), dtype=torch.float64, device="cuda")
    S.loglik_grad(m, S.FP64, y, x, ll, g)
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    S.release_workspace()
    assert torch.cuda.mem_get_info()[0] - kept >= 37 * 3 * P * 8
    S.release_workspace()
    assert _same(torch, _work(S, torch, 21), want)


def test_kept_memory_does_not_refuse_a_context(S):
    """With the device filled up to less than a run's buffers beside what the pool
    keeps, smc_init succeeds (the driver takes unused pool memory back)."""
    torch = torch_cuda()
    K, P, T = 2, 500000, 600          # 444 MB of checkpoints
    truth = egarch_truth(K, 2)
    yh = I.simulate_egarch(truth, T, seed=71)
    y, m = dev(yh), S.model_egarch(K, 2, True)
    x = soa(np.resize(particles(14, truth, K, 2, True, 1000, 5), (P, 14)))
    ll, g = torch.zeros(P, dtype=torch.float64, device="cuda"), torch.zeros((14, P), dtype=torch.float64, device="cuda")
    theta0 = S.draw_prior(m, 1, 1 << 20)
    torch.cuda.synchronize()
    S.release_workspace()
    S.loglik_grad(m, S.FP64, y, x, ll, g)
    torch.cuda.synchronize()
    # a run of 1,048,576 particles needs about 500 MB: leave 300 beside the 444 kept
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        cfg = S.config_default(J=256, N=4096, precision=S.FP32, seed=1)
        ctx = S.init(m, cfg, yh, theta0, theta0_on_device=True)
        del ctx
    finally:
        del fill
        torch.cuda.empty_cache()
