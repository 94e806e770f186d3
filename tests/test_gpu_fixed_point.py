"""FP64 kernels around the edges of the fixed-point recursion: block and chunk
ends, particles that leave its ranges for a block or for good, and proposals
whose likelihood is not carried to the end because they are rejected whatever
it is.  Against the FP64 oracle at the FP64 contract's 1e-9 relative."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_util import dev, egarch_truth, host, particles, soa, torch_cuda
from paper_1304_4334_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch_cuda()
    from paper_1304_4334_gb300 import smc
    return smc


def _series(truth, T):
    y = I.simulate_egarch(truth, T, seed=71)
    y[min(T - 1, 30)] += 3.0       # 300 standard deviations: out of range for one block
    return y


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 2), (3, 4), (4, 3)])
@pytest.mark.parametrize("T", [1, 31, 32, 33, 511, 512, 513, 1025])
@pytest.mark.parametrize("outlier", [False, True])
def test_loglik_block_edges_and_range_exits(S, K, I_, T, outlier):
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = _series(truth, T) if outlier else I.simulate_egarch(truth, T, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    P = 70
    th = particles(spec.d, truth, K, I_, True, P, 73, prior=O.table1_prior(K, I_, True), frac_prior=0.3)
    ll_o, st_o = O.loglik(spec, y, th, with_state=True, nthreads=4)
    ll = torch.empty(P, dtype=torch.float64, device="cuda")
    st = torch.empty((K + 1, P), dtype=torch.float64, device="cuda")
    S.loglik(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(th), ll, None, st)
    ll, st = host(ll), host(st).T
    sane = ll_o > -1e7
    cloud = np.arange(P) >= int(P * 0.3)
    assert cloud[sane].sum() > P // 2
    np.testing.assert_allclose(ll[sane], ll_o[sane], rtol=1e-9)
    # (the oracle forms h_t itself, whose overflow makes its value -inf where log
    # h_t is still finite: those are not compared)
    assert np.all(ll[np.isfinite(ll_o) & ~sane] < -1e6)
    np.testing.assert_allclose(st[sane & cloud], st_o[sane & cloud], rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 3)])
@pytest.mark.parametrize("phi", [0.0, 1e-4, 0.02, 1.0])
def test_mutation_with_out_of_range_proposals(S, K, I_, phi):
    """Prior draws moved with a wide proposal: many recursions explode.  The
    decision, theta, l, log prior and state equal the oracle's."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    T, P = 333, 300
    y = I.simulate_egarch(truth, T, seed=75)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    th = particles(spec.d, truth, K, I_, True, P, 77, prior=O.table1_prior(K, I_, True), frac_prior=0.5)
    ll, st = O.loglik(spec, y, th, with_state=True, nthreads=4)
    keep = ll > -1e7
    th, ll, st = th[keep], ll[keep], st[keep]
    P = len(th)
    lp = O.logprior(spec, th)
    L = np.diag(np.full(spec.d, 0.4))
    th_o, ll_o, lp_o, st_o, acc_o, n_o = O.mutate_rw(spec, y, th.copy(), ll.copy(), lp.copy(), st.copy(), L, phi, 9, 2, 3)
    g = [soa(th), dev(ll), dev(lp), soa(st)]
    n = S.mutate_rw(S.model_egarch(K, I_, True), S.FP64, dev(y), *g, dev(L), phi, 9, 2, 3)
    th_g, ll_g, lp_g, st_g = host(g[0]).T, host(g[1]), host(g[2]), host(g[3]).T
    acc_g = np.any(th_g != th, axis=1)
    acc_o = np.any(th_o != th, axis=1)
    assert n == n_o and np.array_equal(acc_g, acc_o), (n, n_o)
    assert 0 < acc_o.sum() < P
    sane = ll_o > -1e7
    np.testing.assert_allclose(ll_g[sane], ll_o[sane], rtol=1e-9)
    np.testing.assert_allclose(th_g, th_o, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(lp_g, lp_o, rtol=1e-12)
    assert np.all(ll_g[np.isfinite(ll_o) & ~sane] < -1e6)


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 2), (3, 4)])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 130])
def test_gradient_with_range_exits(S, K, I_, T):
    """Segment edges, a shock out of range, and parameters out of range (a
    component far narrower than its distance from zero, a large beta), against
    the oracle's gradient at the FP64 gradient's 1e-7 of the largest entry."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = _series(truth, T)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    P = 48
    th = particles(spec.d, truth, K, I_, True, P, 79)
    if I_ > 1:
        th[:8, spec.d - 1] = -4.0                  # sigma of the last component
        th[:8, spec.d - I_ - 1] = 3.0              # and its mean
    th[8:12, 2 + K] = np.log(1.5)                  # beta_1
    ll_o, g_o = O.loglik_grad(spec, y, th)
    ll = torch.empty(P, dtype=torch.float64, device="cuda")
    g = torch.empty((spec.d, P), dtype=torch.float64, device="cuda")
    S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(th), ll, g)
    ll, g = host(ll), host(g).T
    sane = (ll_o > -1e7) & np.isfinite(g_o).all(axis=1)   # (an overflow on the way leaves the oracle's NaN)
    assert sane[12:].sum() > 30
    np.testing.assert_allclose(ll[sane], ll_o[sane], rtol=1e-9)
    err = np.abs(g - g_o)[sane].max(axis=1) / np.abs(g_o[sane]).max(axis=1)
    assert err.max() <= 1e-7, err.max()


@pytest.mark.parametrize("K,I_", [(1, 2), (2, 3), (4, 4)])
@pytest.mark.parametrize("T", [1, 16, 17, 33, 530])
def test_gradient_kernels_of_few_and_many_particles(S, K, I_, T):
    """The same particles in a call small enough for two warps per 32 of them and
    in one that is not, a ragged last warp, range exits and a shock out of range
    included: two orders of the same FP64 sums, so far within 1e-9 (of the
    largest entry of the gradient, whose entries cancel)."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = _series(truth, T)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    P, n = 77, 200 * torch.cuda.get_device_properties(0).multi_processor_count
    th = particles(spec.d, truth, K, I_, True, P, 81, prior=O.table1_prior(K, I_, True), frac_prior=0.2)
    th[:8, spec.d - 1] = -4.0                      # a component far narrower
    th[:8, spec.d - I_ - 1] = 3.0                  # than its distance from zero
    out = []
    for tt in (th, np.resize(th, (n, spec.d))):
        ll = torch.empty(len(tt), dtype=torch.float64, device="cuda")
        g = torch.empty((spec.d, len(tt)), dtype=torch.float64, device="cuda")
        st = torch.empty((K + 1, len(tt)), dtype=torch.float64, device="cuda")
        S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(tt), ll, g, st)
        out.append([host(ll)[:P], host(g).T[:P], host(st).T[:P]])
    (l1, g1, s1), (l2, g2, s2) = out
    assert np.array_equal(l1 > -1e7, l2 > -1e7)
    sane = (l2 > -1e7) & np.isfinite(g2).all(axis=1)
    assert sane.sum() > P // 2
    np.testing.assert_allclose(l1[sane], l2[sane], rtol=1e-9)
    assert (np.abs(g1 - g2)[sane].max(axis=1) <= 1e-9 * np.abs(g2[sane]).max(axis=1)).all()
    np.testing.assert_allclose(s1[sane], s2[sane], rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("K,I_", [(1, 2), (2, 3), (4, 4)])
@pytest.mark.parametrize("T", [1, 31, 32, 33, 65, 530])
def test_likelihood_kernels_of_few_and_many_particles(S, K, I_, T):
    """As above for the log likelihood: two or three warps per 32 particles in
    the small call, one in the large, the same integer sums but for the order of
    the mixture sums' product and the FP64 parts of range exits."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = _series(truth, T)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    P, n = 77, 200 * torch.cuda.get_device_properties(0).multi_processor_count
    th = particles(spec.d, truth, K, I_, True, P, 83, prior=O.table1_prior(K, I_, True), frac_prior=0.2)
    th[:8, spec.d - 1] = -4.0                      # a component far narrower
    th[:8, spec.d - I_ - 1] = 3.0                  # than its distance from zero
    out = []
    for tt in (th, np.resize(th, (n, spec.d))):
        ll = torch.empty(len(tt), dtype=torch.float64, device="cuda")
        lp = torch.empty(len(tt), dtype=torch.float64, device="cuda")
        st = torch.empty((K + 1, len(tt)), dtype=torch.float64, device="cuda")
        S.loglik(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(tt), ll, lp, st)
        out.append([host(ll)[:P], host(lp)[:P], host(st).T[:P]])
    (l1, p1, s1), (l2, p2, s2) = out
    assert np.array_equal(l1 > -1e7, l2 > -1e7) and np.array_equal(p1, p2)
    sane = l2 > -1e7
    assert sane.sum() > P // 2
    np.testing.assert_allclose(l1[sane], l2[sane], rtol=1e-9)
    np.testing.assert_allclose(s1[sane], s2[sane], rtol=1e-9, atol=1e-12)


def _few_and_many(S, K, I_, spec, y, th, grad):
    """Likelihoods (and gradients) of the same particles from the kernels of a
    small call and of a large one."""
    torch = torch_cuda()
    n = 200 * torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for tt in (th, np.resize(th, (n, spec.d))):
        ll = torch.empty(len(tt), dtype=torch.float64, device="cuda")
        st = torch.empty((K + 1, len(tt)), dtype=torch.float64, device="cuda")
        if grad:
            g = torch.empty((spec.d, len(tt)), dtype=torch.float64, device="cuda")
            S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(tt), ll, g, st)
        else:
            S.loglik(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(tt), ll, None, st)
        out.append(host(ll)[:len(th)])
    return out


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 2), (3, 4)])
@pytest.mark.parametrize("grad", [False, True])
def test_parameters_that_are_not_finite(S, K, I_, grad):
    """Each parameter in turn NaN, inf or -inf: the log likelihood is the
    oracle's, -inf for every NaN, in every kernel."""
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 100, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    values = [np.nan, np.inf, -np.inf]
    th = np.repeat(particles(spec.d, truth, K, I_, True, 1, 85), 3 * spec.d, axis=0)
    for j in range(spec.d):
        th[3 * j:3 * j + 3, j] = values
    ll_o = O.loglik(spec, y, th)
    assert np.all(ll_o[::3] == -np.inf)
    for ll in _few_and_many(S, K, I_, spec, y, th, grad):
        assert np.all(ll[::3] == -np.inf), np.flatnonzero(ll[::3] != -np.inf)
        np.testing.assert_allclose(ll[np.isfinite(ll_o)], ll_o[np.isfinite(ll_o)], rtol=1e-9)
        assert np.all(ll[~np.isfinite(ll_o)] == -np.inf)


@pytest.mark.parametrize("K,I_", [(1, 2), (2, 2), (3, 4)])
@pytest.mark.parametrize("grad", [False, True])
def test_mixture_parameters_past_the_exponentials_range(S, K, I_, grad):
    """Each mixture parameter in turn at +-400 and +-800, where its exponential
    or the component's standard deviation under- or overflows: a component with
    sigma_i = 0 has a density that is NaN, and so -inf, whichever its place."""
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 100, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    values = [-800.0, -400.0, 400.0, 800.0]
    th = np.repeat(particles(spec.d, truth, K, I_, True, 1, 87), 4 * 3 * I_, axis=0)
    for j in range(3 * I_):
        th[4 * j:4 * j + 4, spec.d - 3 * I_ + j] = values
    ll_o = O.loglik(spec, y, th)
    sane = ll_o > -1e7
    assert np.all(ll_o[4 * 2 * I_::4] == -np.inf)      # sigma_i = exp(-800)
    for ll in _few_and_many(S, K, I_, spec, y, th, grad):
        np.testing.assert_allclose(ll[sane], ll_o[sane], rtol=1e-9)
        assert np.all(ll[~sane] < -1e6), np.flatnonzero(~(ll < -1e6) & ~sane)


def _gradient64(th, y, K, I_):
    """The gradient by torch in FP64, with p_i = 2 / (1 + exp(-2 theta_i)) free of
    cancellation (the oracle's 1 + tanh(theta_i) loses a small p_i's digits)."""
    torch = torch_cuda()
    t = torch.tensor(th.T.copy(), requires_grad=True)
    j = 2 + 3 * K
    al, be, ga = torch.tanh(t[2:2 + K]), torch.exp(t[2 + K:2 + 2 * K]), t[2 + 2 * K:j]
    p = 2.0 / (1.0 + torch.exp(-2.0 * t[j:j + I_]))
    p = p / p.sum(0)
    mu, s = t[j + I_:j + 2 * I_], torch.exp(t[j + 2 * I_:])
    mu = mu - (p * mu).sum(0)
    c = 1.0 / torch.sqrt((p * (mu * mu + s * s)).sum(0))
    lp, m, a = torch.log(p) - torch.log(c * s), c * mu, 1.0 / (c * s)
    v, ll = torch.zeros_like(al), 0.0
    for n, yt in enumerate(y):
        if n:
            v = al * v + be * (e.abs() - np.sqrt(2.0 / np.pi)) + ga * e
        lh = t[1] + 0.5 * v.sum(0)
        e = (float(yt) - t[0] / 1000.0) * torch.exp(-lh)
        z = (e - m) * a
        ll = ll + torch.logsumexp(lp - 0.5 * z * z, 0) - lh
    (g,) = torch.autograd.grad(ll.sum(), t)
    return g.numpy().T


@pytest.mark.parametrize("K,I_", [(1, 2), (2, 3), (4, 4)])
@pytest.mark.parametrize("theta_p", [-6.0, -12.0, -15.0])
def test_gradient_of_a_rare_component(S, K, I_, theta_p):
    """A last component of probability about 6e-6, 4e-11, 1e-13: its parameters'
    gradients are as small, and as accurate for their size (1e-9; FP64 leaves
    1e-12) as the others', in both gradient kernels."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 130, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    th = particles(spec.d, truth, K, I_, True, 40, 89)
    th[:, spec.d - 2 * I_ - 1] = theta_p
    want = _gradient64(th, y, K, I_)
    last = [spec.d - 2 * I_ - 1, spec.d - I_ - 1, spec.d - 1]
    for n in (40, 200 * torch.cuda.get_device_properties(0).multi_processor_count):
        x = np.resize(th, (n, spec.d))
        ll = torch.empty(n, dtype=torch.float64, device="cuda")
        g = torch.empty((spec.d, n), dtype=torch.float64, device="cuda")
        S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(x), ll, g)
        np.testing.assert_allclose(host(g)[last, :40].T, want[:, last], rtol=1e-9)


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 2), (3, 4)])
@pytest.mark.parametrize("grad", [False, True])
def test_end_state_of_a_tiny_shock(S, K, I_, grad):
    """A last return within 2^-40 of the mean leaves a shock of 1e-14 or so, which
    the recursion itself carries in units of 2^-53: the state given out is the
    shock as FP64 has it."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 45, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    th = particles(spec.d, truth, K, I_, True, 70, 101)
    th[:, 0] = th[0, 0]
    y[-1] = th[0, 0] / 1000.0 * (1.0 + 2.0 ** -40)
    ll_o, st_o = O.loglik(spec, y, th, with_state=True)
    assert np.all(np.abs(st_o[:, K]) < 1e-12) and np.all(st_o[:, K] != 0.0)
    for n in (70, 200 * torch.cuda.get_device_properties(0).multi_processor_count):
        x = np.resize(th, (n, spec.d))
        ll = torch.empty(n, dtype=torch.float64, device="cuda")
        st = torch.empty((K + 1, n), dtype=torch.float64, device="cuda")
        if grad:
            g = torch.empty((spec.d, n), dtype=torch.float64, device="cuda")
            S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(x), ll, g, st)
        else:
            S.loglik(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(x), ll, None, st)
        np.testing.assert_allclose(host(st)[K, :70], st_o[:, K], rtol=1e-9)


@pytest.mark.parametrize("K,I_", [(1, 1), (2, 3)])
def test_mutation_leaves_the_likelihoods_state(S, K, I_):
    """The state of accepted proposals, tiny last shock included, is the one that
    the likelihood gives at the new parameters, to the bit."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 45, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    P = 150 * torch.cuda.get_device_properties(0).multi_processor_count
    th = particles(spec.d, truth, K, I_, True, P, 103)
    th[:, 0] = th[0, 0]
    y[-1] = th[0, 0] / 1000.0 * (1.0 - 2.0 ** -40)
    L = np.diag(np.full(spec.d, 0.02))
    L[0, 0] = 0.0
    m, x, obs = S.model_egarch(K, I_, True), soa(th), dev(y)
    ll, lp = (torch.empty(P, dtype=torch.float64, device="cuda") for _ in range(2))
    st = torch.empty((K + 1, P), dtype=torch.float64, device="cuda")
    S.loglik(m, S.FP64, obs, x, ll, lp, st)
    assert 0 < S.mutate_rw(m, S.FP64, obs, x, ll, lp, st, dev(L), 0.5, 9, 2, 3) < P
    ll2, lp2, st2 = torch.empty_like(ll), torch.empty_like(lp), torch.empty_like(st)
    S.loglik(m, S.FP64, obs, x, ll2, lp2, st2)
    assert torch.equal(ll, ll2) and torch.equal(st, st2) and bool((st[K] != 0).all())


@pytest.mark.parametrize("K,I_", [(1, 1), (1, 2), (3, 4)])
@pytest.mark.parametrize("side", [-1.0, 1.0])
def test_gradient_at_a_shock_below_the_fixed_point_unit(S, K, I_, side):
    """A return one rounding off the mean: the shock (5e-18) is not zero, and the
    derivative of |eps| there has its sign."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 45, seed=71)
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    th = particles(spec.d, truth, K, I_, True, 40, 105)
    th[:, 0] = th[0, 0]
    y[20] = np.nextafter(th[0, 0] / 1000.0, side)
    ll_o, g_o = O.loglik_grad(spec, y, th)
    for n in (40, 200 * torch.cuda.get_device_properties(0).multi_processor_count):
        ll = torch.empty(n, dtype=torch.float64, device="cuda")
        g = torch.empty((spec.d, n), dtype=torch.float64, device="cuda")
        S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(np.resize(th, (n, spec.d))), ll, g)
        err = np.abs(host(g)[:, :40].T - g_o).max(axis=1) / np.abs(g_o).max(axis=1)
        assert err.max() <= 1e-7, err.max()


@pytest.mark.parametrize("K,I_", [(1, 2), (2, 3)])
def test_gradient_of_an_enormous_shock(S, K, I_):
    """A return of 1e140: l is about -1e283, finite, and so is its gradient, in
    both gradient kernels (nothing is scaled on the way)."""
    torch = torch_cuda()
    truth = egarch_truth(K, I_)
    y = I.simulate_egarch(truth, 40, seed=71)
    y[-1] = 1e140
    spec = O.ModelSpec(K=K, I=I_, gamma=True)
    th = particles(spec.d, truth, K, I_, True, 40, 107)
    ll_o, g_o = O.loglik_grad(spec, y, th)
    assert np.isfinite(ll_o).all() and np.isfinite(g_o).all()
    for n in (40, 200 * torch.cuda.get_device_properties(0).multi_processor_count):
        ll = torch.empty(n, dtype=torch.float64, device="cuda")
        g = torch.empty((spec.d, n), dtype=torch.float64, device="cuda")
        S.loglik_grad(S.model_egarch(K, I_, True), S.FP64, dev(y), soa(np.resize(th, (n, spec.d))), ll, g)
        np.testing.assert_allclose(host(ll)[:40], ll_o, rtol=1e-9)
        err = np.abs(host(g)[:, :40].T - g_o).max(axis=1) / np.abs(g_o).max(axis=1)
        assert err.max() <= 1e-7, err.max()
