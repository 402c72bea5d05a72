"""Launch shapes at the edges of their ranges: tiles with remainders, the
smallest sizes, every branch of a size rule."""
import math

import numpy as np
import pytest
import torch

from gpu_util import angle_diff, ensure_built, kur_run
from paper_0903_3852_gb300 import inputs, sde

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,R", [(1, 1), (7, 2), (33, 1), (1000, 3), (1025, 2), (1024, 40), (129, 500), (2047, 60)])
@pytest.mark.parametrize("euler", [False, True])
def test_pairwise_shapes_match_mean_field(N, R, euler):
    """Five steps of the all-pairs sum against the mean-field form (SRK2) or the
    direct coupling sums (Euler).  A step's coupling differs by at most a few
    1e-7 N terms times K dt / N = 1e-8 rad, phases are kept to 1.5e-9 rad and
    returned in FP32 (half an ulp at 2 pi: 2.4e-7): 1e-6 holds all of them."""
    ensure_built()
    w = inputs.kuramoto_uniform(n_osc=N, replicas=R, seed=N)
    kw = dict(K=2.0, D=0.05, dt=0.01, seed=3, sample_every=2)
    flags = sde.SDE_FLAG_EULER if euler else 0
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, R, flags=flags, **kw)
    if euler:
        phi, _, _ = kur_run(ens, w["phi0"], w["omega"], 0, 1)
        ref = ens.coupling(torch.from_numpy(w["phi0"]).cuda()).cpu().numpy().astype(np.float64)
        srk = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, R, **dict(kw, K=0.0))
        free, _, _ = kur_run(srk, w["phi0"], w["omega"], 0, 1)  # without coupling both schemes are one
        assert np.abs(angle_diff(phi, free + 0.01 * ref)).max() <= 1e-6
        return
    phi, r, _ = kur_run(ens, w["phi0"], w["omega"], 0, 5)
    mf = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_MEANFIELD, N, R, **kw)
    phi_mf, r_mf, _ = kur_run(mf, w["phi0"], w["omega"], 0, 5)
    assert np.abs(angle_diff(phi, phi_mf)).max() <= 1e-6
    assert np.abs(r - r_mf).max() <= 2e-5


@pytest.mark.parametrize("N,R", [(1, 3), (3, 5), (5, 2), (1023, 3), (4098, 2)])
@pytest.mark.parametrize("shift", [0, 1])
def test_grid_wide_chunks_match_replica_form(N, R, shift):
    """The grid-wide mean field's 16-byte chunks where replicas start inside one,
    and frequencies that start off a 16-byte boundary, against one CTA per
    replica over steps 3 .. 9.  The replica form's sums are within N 2^-18, K dt / N
    times that is 8e-8 per step, and phases come back in FP32 (2.4e-7): 1e-6."""
    ensure_built()
    w = inputs.kuramoto_uniform(n_osc=N, replicas=R, seed=N)
    phi0 = torch.from_numpy(w["phi0"]).cuda()
    store = torch.zeros(N * R + shift, device="cuda")
    omega = store[shift:].view(R, N)
    omega.copy_(torch.from_numpy(w["omega"]))
    got = []
    for kw in (dict(schedule=sde.SDE_SCHED_GRID), dict(cluster_ctas=1)):
        ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_MEANFIELD, N, R, 2.0, 0.05, 0.01, 3, sample_every=2, **kw)
        phi, r = torch.empty_like(phi0), torch.empty((4, R), dtype=torch.float64, device="cuda")
        ens.run_kuramoto(3, 9, phi0, phi, omega, r)
        got.append((phi.cpu().numpy().astype(np.float64), r.cpu().numpy()))
    assert np.abs(angle_diff(got[0][0], got[1][0])).max() <= 1e-6
    assert np.abs(got[0][1] - got[1][1]).max() <= 2e-5


@pytest.mark.parametrize("N,R", [(1, 1), (2, 3), (129, 9), (512, 1), (513, 20), (1023, 2), (2000, 4)])
@pytest.mark.parametrize("euler", [False, True])
def test_pairwise_cluster_form_resumes(N, R, euler):
    """A replica per cluster, at the edges of its groups of receivers and rounds of
    sources: steps 3 .. 10 in one run and in two (the phases return in FP32
    between them: 2.4e-7, grown by at most 1 + K dt per step), and against the
    mean-field form with the bound above."""
    ensure_built()
    w = inputs.kuramoto_uniform(n_osc=N, replicas=R, seed=N)
    kw = dict(K=2.0, D=0.05, dt=0.01, seed=3, sample_every=3)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, R, flags=sde.SDE_FLAG_EULER if euler else 0, **kw)
    assert ens.tuning()[0] == 512 and ens.tuning()[1] == 1  # the cluster form
    phi, r, _ = kur_run(ens, w["phi0"], w["omega"], 3, 10)
    half, _, _ = kur_run(ens, w["phi0"], w["omega"], 3, 6)
    two, _, _ = kur_run(ens, half.astype(np.float32), w["omega"], 6, 10)
    assert np.abs(angle_diff(phi, two)).max() <= 1e-6
    if not euler:
        mf = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_MEANFIELD, N, R, **kw)
        phi_mf, r_mf, _ = kur_run(mf, w["phi0"], w["omega"], 3, 10)
        assert np.abs(angle_diff(phi, phi_mf)).max() <= 1e-6
        assert np.abs(r - r_mf).max() <= 2e-5


@pytest.mark.parametrize("N,R", [(8, 1), (16, 3), (136, 13), (264, 25), (512, 100), (1000, 7), (3000, 28)])
def test_fp32_gemm_shapes(N, R):
    """Coupling sums of the FP32 form against FP64: every chain of N FMAs errs by
    at most N 2^-24 sum|K_ij| (the sines by 2^-23 each)."""
    ensure_built()
    w = inputs.kuramoto_general(n_osc=N, replicas=R, seed=N)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_GENERAL_FP32, N, R, 0.0, 0.02, 0.005, 1)
    K = torch.from_numpy(w["Kmat"]).cuda()
    ens.set_coupling(K)
    phi = torch.from_numpy(w["phi0"]).cuda()
    got = ens.coupling(phi).double()
    x, Kt = phi.double(), K.double().t()
    s, c = torch.sin(x), torch.cos(x)
    ref = c * (s @ Kt) - s * (c @ Kt)
    bound = 2.0 * (N + 8) * 2.0 ** -24 * K.double().abs().sum(1)
    assert torch.all((got - ref).abs() <= bound)


@pytest.mark.parametrize("hidden,n_hidden,n_in,B,max_batch", [
    (64, 1, 1, 1, 1), (256, 3, 5, 63, 64), (256, 3, 5, 65, 4096), (320, 2, 8, 129, 129), (256, 2, 7, 20000, 20000)])
def test_members_train_together_as_alone(hidden, n_hidden, n_in, B, max_batch):
    """Members share launches (in groups where their batches fill the activation
    rows: the last case): each ends bit for bit where it ends alone."""
    ensure_built()
    rng = np.random.default_rng(B)
    M = 3
    X = torch.from_numpy(rng.uniform(-1, 1, (M, B, n_in)).astype(np.float32)).cuda()
    y = torch.sin(2 * X[..., 0]).contiguous()
    kw = dict(n_in=n_in, hidden=hidden, n_hidden=n_hidden, max_batch=max_batch)
    both = sde.Mlp(members=M, seed=5, **kw)
    alone = []
    for q in range(M):
        m = sde.Mlp(members=1, seed=1, **kw)
        m.set_params(0, both.get_params(q))
        alone.append(m)
    loss = torch.zeros(M, device="cuda")
    for _ in range(2):
        both.train_step_members(X, y, loss)
        for q, m in enumerate(alone):
            l1 = torch.zeros(1, device="cuda")
            m.train_step(X[q].contiguous(), y[q].contiguous(), l1)
            assert l1.item() == loss[q].item() and math.isfinite(l1.item())
    for q, m in enumerate(alone):
        assert torch.equal(both.get_params(q), m.get_params(0))


FIG2 = dict(gamma=0.9, a=4.2, omega=4.9, f=0.1, D=1e-3)


def _josephson(points, paths, steps, P, windows, x0, v0, flags=0, **kw):
    n = int(np.sum(paths))
    ens = sde.Ensemble.josephson(points, paths, steps, 7, steps_per_period=P, flags=flags, **kw)
    x, v = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    w = torch.empty(n, dtype=torch.int32, device="cuda")
    vs = torch.empty(n, dtype=torch.float64, device="cuda")
    xin, vin, more, n0 = x0, v0, {}, 0
    for n1 in windows:
        ens.run_josephson(n0, n1, xin, vin, x, v, w, vs, **more)
        xin, vin, more, n0 = x, v, dict(w_in=w, vsum_in=vs), n1
    return ens.tuning()[1], (x, v, w, vs), ens.observables()


@pytest.mark.parametrize("paths,steps,P,windows,flags,v_scale", [
    ([1024], [1000], 200, [1000], 0, 2.0),
    ([1], [5], 200, [1, 3, 5], 0, 2.0),  # inside one group of four steps
    ([100, 33, 64], [997, 1501, 64], 100, [63, 64, 65, 502, 1600], 0, 2.0),  # windows and their starts inside groups
    ([70, 31], [400, 258], 200, [399, 400], sde.SDE_FLAG_EULER, 2.0),
    ([96], [300], 1020, [300], 0, 2.0),  # the longest per-warp drive table
    ([64], [200], 200, [200], 0, 60.0)])  # velocities beyond the block path's bound
def test_small_ensembles_equal_the_one_warp_kernels(paths, steps, P, windows, flags, v_scale):
    """The kernel of small ensembles (steps and noise in different warps) against
    two paths per thread: states and window sums bit for bit, through the
    allocation-free entry point as well; observables to rounding."""
    ensure_built()
    n = int(np.sum(paths))
    rng = np.random.default_rng(n)
    x0 = torch.from_numpy(rng.uniform(-1, 2, n).astype(np.float32)).cuda()
    v0 = torch.from_numpy(rng.uniform(-v_scale, v_scale, n).astype(np.float32)).cuda()
    points = [dict(FIG2, f=0.05 * i, D=1e-4 * 5 ** i) for i in range(len(paths))]
    variant, a, obs_a = _josephson(points, paths, steps, P, windows, x0, v0, flags)
    assert variant == 21
    _, b, obs_b = _josephson(points, paths, steps, P, windows, x0, v0, flags, block_threads=128, paths_per_thread=2)
    assert all(torch.equal(p, q) for p, q in zip(a, b))
    assert np.allclose(obs_a["mean"], obs_b["mean"], rtol=1e-12, atol=1e-14)
    assert np.allclose(obs_a["var"], obs_b["var"], rtol=1e-10, atol=1e-14)


@pytest.mark.parametrize("n,P,steps", [(1, 200, 10), (333, 100, 130), (40000, 200, 66), (45000, 7, 33),
                                       (400000, 200, 21)])
def test_noalloc_kernels_equal_the_plain_schedule(n, P, steps):
    """Every kernel of the allocation-free entry point (pairs of warps, two and
    four paths per thread) against one path per thread, bit for bit."""
    ensure_built()
    rng = np.random.default_rng(n)
    x0 = torch.from_numpy(rng.random(n).astype(np.float32)).cuda()
    v0 = torch.from_numpy(rng.uniform(-2, 2, n).astype(np.float32)).cuda()
    _, a, obs = _josephson([FIG2], [n], [steps], P, [steps], x0, v0, schedule=sde.SDE_SCHED_PLAIN, block_threads=256,
                           paths_per_thread=1)
    x, v, w, vs = (torch.empty_like(t) for t in a)
    row = torch.empty(5, dtype=torch.float64, device="cuda")
    sde.josephson_run_noalloc(FIG2, P, n, steps, 7, 0, steps, x0, v0, x, v, w, vs, row)
    assert all(torch.equal(p, q) for p, q in zip(a, (x, v, w, vs)))
    got = row.cpu().numpy()
    assert np.allclose(got, [obs[k][0] for k in ("mean", "var", "se", "count", "t")], rtol=1e-10, atol=1e-14)


@pytest.mark.parametrize("n,steps", [(1, 3), (65, 9), (5000, 40), (80000, 10)])
def test_fp64_block_sizes(n, steps):
    """Every block size of the FP64 kernel and windows inside a group of four
    steps, against torch in FP64 (same Philox words through the library):
    rounding of ~30 operations per step on values below ~10, 40 steps."""
    ensure_built()
    P, pt = 100, dict(FIG2, gamma=3.0)
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.random(n)).cuda()
    v = torch.from_numpy(rng.uniform(-2, 2, n)).cuda()
    xo, vo, so = torch.empty_like(x), torch.empty_like(v), torch.empty_like(v)
    sde.josephson_run_fp64(pt, P, steps, 5, 0, steps, x, v, xo, vo, vsum_out=so, point_index=2)
    dt = 2 * math.pi / (pt["omega"] * P)
    s, vsum = math.sqrt(2 * pt["gamma"] * pt["D"] * dt), torch.zeros_like(v)
    ctr = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
    ctr[:, 1], ctr[:, 2], ctr[:, 3] = torch.arange(n, device="cuda"), 2, 1

    def force(x, v, k):
        return -pt["gamma"] * v - 2 * math.pi * torch.cos(2 * math.pi * x) + pt["a"] * math.cos(
            2 * math.pi * (k % P) / P) + pt["f"]

    for k in range(steps):
        if k % 4 == 0:
            ctr[:, 0] = k // 4
            u = (((sde.philox4x32_10(ctr, 5).long() & 0xFFFFFFFF) >> 8) + 1).double() * 2.0 ** -24
            z = []
            for a, b in ((u[:, 0], u[:, 1]), (u[:, 2], u[:, 3])):
                rho = torch.sqrt(-2 * torch.log(a))
                z += [rho * torch.cos(2 * math.pi * b), rho * torch.sin(2 * math.pi * b)]
        noise = s * z[k % 4]
        F1 = force(x, v, k)
        vt = v + dt * F1 + noise
        F2 = force(x + dt * v, vt, k + 1)
        x, v = x + 0.5 * dt * (v + vt), v + 0.5 * dt * (F1 + F2) + noise
        if k + 1 > steps - steps // 2:
            vsum = vsum + v
    for got, ref in ((xo, x), (vo, v), (so, vsum)):
        assert (got - ref).abs().max().item() <= 1e-12


@pytest.mark.parametrize("members,n_hidden,n_in", [(1, 2, 1), (4, 3, 5), (3, 8, 8)])
@pytest.mark.parametrize("B", [1, 128, 129, 6500, 39000])
def test_forward_tiles_are_independent(members, n_hidden, n_in, B):
    """Tensor-core forward with one tile, a ragged tile, one and several tiles
    per CTA (an odd and an even number): every point's result is that of a
    one-tile call bit for bit."""
    ensure_built()
    m = sde.Mlp(n_in=n_in, n_hidden=n_hidden, members=members, max_batch=40000, seed=9)
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    X = torch.rand((B, n_in), generator=g, device="cuda") * 2 - 1
    mean, spread = m.forward(X)
    m.check()
    for b0 in sorted({0, 64 * (B // 128), 128 * (B // 256), max(0, B - 100)}):
        part = X[b0:b0 + 100].contiguous()
        mp, sp = m.forward(part)
        assert torch.equal(mean[b0:b0 + 100], mp) and torch.equal(spread[b0:b0 + 100], sp)
    m.use_tensor_cores(False)
    ref, _ = m.forward(X)
    assert (mean - ref).abs().max().item() <= 2e-3 * max(1.0, ref.abs().max().item())


def _turns_step(th, K, omega, dt, euler):
    """One step without noise on fixed-point phases, the sums in FP64."""
    def drift(t):
        d = (t[:, None, :] - t[:, :, None] + 2 ** 31) % 2 ** 32 - 2 ** 31
        return omega * dt / (2 * np.pi) + K * dt / (2 * np.pi) * np.sin(2 * np.pi / 2 ** 32 * d).mean(2)

    def add(t, d):
        return (t + np.rint(d * 2.0 ** 32).astype(np.int64)) % 2 ** 32

    d1 = drift(th)
    return add(th, d1) if euler else add(th, 0.5 * (d1 + drift(add(th, d1))))


@pytest.mark.parametrize("N,R", [(1000, 3), (1024, 60), (2500, 1), (300, 400)])
@pytest.mark.parametrize("euler", [False, True])
@pytest.mark.parametrize("spread", [0.0, 1e-5])
def test_pairwise_terms_of_a_population_in_step(N, R, euler, spread):
    """Phases within `spread` of one another, strong coupling and a common
    frequency, one SRK2 or two Euler steps: the coupling per source, as read off
    the result, is within 8e-9 of the FP64 sums.  Its parts: the phases come back
    in FP32 (6e-8 below 2 rad, over K dt = 50: 1.2e-9), a fixed-point unit of the
    first stage grown by the second (1.5e-9 K dt, over K dt), and the sums' own
    rounding, 6e-8 of sines below the frame's lag (0.05 rad) and the spread
    (3e-9).  A population wholly in step turns by the same number of units
    everywhere."""
    ensure_built()
    K, dt, omega, steps = 5000.0, 0.01, 5.0, 2 if euler else 1
    rng = np.random.default_rng(N)
    phi0 = (1.0 + spread * rng.uniform(-1, 1, (R, N))).astype(np.float32)
    om = np.full((R, N), omega, np.float32)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, R, K, 0.0, dt, 3, sample_every=1,
                                flags=sde.SDE_FLAG_EULER if euler else 0)
    phi, _, _ = kur_run(ens, phi0, om, 0, steps)
    if spread == 0.0:
        assert (phi == phi[0, 0]).all()
    th = np.rint(phi0[:2].astype(np.float64) / (2 * np.pi) * 2 ** 32).astype(np.int64)
    for _ in range(steps):
        th = _turns_step(th, K, omega, dt, euler)
    err = np.abs(angle_diff(phi[:2], th * (2 * np.pi / 2 ** 32))).max() / (K * dt)
    print("N=%d R=%d euler=%d spread %g: %.2e per source" % (N, R, euler, spread, err))
    assert err <= 8e-9


@pytest.mark.parametrize("N,R", [(1, 3000), (8, 1000), (31, 1500), (32, 900), (33, 900)])
@pytest.mark.parametrize("euler", [False, True])
def test_pairwise_many_small_replicas(N, R, euler):
    """A warp per replica up to 32 oscillators, and one more: the bounds of
    test_pairwise_shapes_match_mean_field."""
    test_pairwise_shapes_match_mean_field(N, R, euler)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, R, 2.0, 0.05, 0.01, 3,
                                flags=sde.SDE_FLAG_EULER if euler else 0)
    assert (ens.tuning()[:2] == (32, 1)) == (N <= 32)


@pytest.mark.parametrize("N,block,cluster,flags,opt", [
    (700, 256, 1, 0, 3), (600, 128, 1, 0, 5), (750, 128, 1, 0, 6), (1400, 256, 2, 0, 3), (2399, 128, 4, 0, 5),
    (3000, 128, 4, 0, 6), (4600, 128, 8, 0, 5), (1400, 256, 2, sde.SDE_FLAG_ASYNC_EXCHANGE, 3),
    (2399, 128, 4, sde.SDE_FLAG_ASYNC_EXCHANGE, 5), (3000, 128, 4, sde.SDE_FLAG_ASYNC_EXCHANGE, 6),
    (4600, 128, 8, sde.SDE_FLAG_ASYNC_EXCHANGE, 5)])
def test_odd_counts_per_thread_equal_a_power_of_two(N, block, cluster, flags, opt):
    """The mean field with 3, 5 and 6 oscillators per thread against 8 or 16 in one
    CTA: the sums are exact integers, so phases and r(t) agree bit for bit."""
    ensure_built()
    w = inputs.kuramoto_uniform(n_osc=N, replicas=3, seed=N)
    kw = dict(K=2.0, D=0.05, dt=0.01, seed=3, sample_every=3)
    got = []
    for shape in (dict(block_threads=block, cluster_ctas=cluster, flags=flags),
                  dict(block_threads=(-(-N // 16) + 31) // 32 * 32, cluster_ctas=1)):
        ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_MEANFIELD, N, 3, **kw, **shape)
        got.append((ens.tuning(), *kur_run(ens, w["phi0"], w["omega"], 2, 13)[:2]))
    assert got[0][0][:2] == (block, opt) and got[1][0][1] in (8, 16)
    assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][2], got[1][2])


@pytest.mark.parametrize("shift_in,shift_out", [(0, 0), (1, 0), (0, 3), (2, 1)])
def test_phases_of_any_range_and_alignment(shift_in, shift_out):
    """A run of no steps returns every phase reduced to [0, 2 pi): the fixed-point
    turns are those of the FP64 quotient within one unit (2^-32 turn), the result
    their FP32 rounding (2.4e-7 below 2 pi, one unit 1.5e-9)."""
    ensure_built()
    rng = np.random.default_rng(5)
    phi = np.concatenate([rng.uniform(0, 8, 20000), rng.uniform(-60, 60, 20000), rng.uniform(-1e-9, 1e-9, 200),
                          [0.0, -0.0, 1e-30, 1e-12, -1e-12, 3.0, 6.2831850, 6.2831855, 7.9999995, 8.0, -8.0, 1e4, -1e4,
                           1e7]]).astype(np.float32)
    phi = np.concatenate([phi, phi[: 3 - phi.size % 4]])  # not a multiple of four
    N = phi.size
    src, dst = torch.zeros(N + shift_in, device="cuda"), torch.full((N + shift_out + 1,), -1.0, device="cuda")
    src[shift_in:] = torch.from_numpy(phi)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_PAIRWISE, N, 1, 1.0, 0.0, 0.01, 1, sample_every=0)
    omega = torch.zeros(N, device="cuda")
    ens.run_kuramoto(4, 4, src[shift_in:].view(1, N), dst[shift_out:shift_out + N].view(1, N), omega.view(1, N))
    out = dst.cpu().numpy().astype(np.float64)
    assert (out[:shift_out] == -1).all() and out[-1] == -1
    out = out[shift_out:shift_out + N]
    t = phi.astype(np.float64) / (2 * np.pi)
    ref = (t - np.floor(t)) * (2 * np.pi)
    assert out.min() >= 0.0 and out.max() <= np.float32(2 * np.pi)
    assert np.abs(angle_diff(out, ref)).max() <= 2.4e-7 + 1.5e-9
    near = np.abs(phi) < 1e-3
    assert np.abs(angle_diff(out[near & (phi >= 0)], ref[near & (phi >= 0)])).max() <= 1.5e-9


@pytest.mark.parametrize("N,R,tn", [(8, 3, 1), (136, 7, 1), (264, 64, 2), (520, 33, 2), (512, 100, 3), (1000, 33, 3),
                                    (264, 200, 5), (512, 400, 7), (2000, 25, 7), (1496, 64, 8)])
def test_fp32_gemm_errs_like_fp32(N, R, tn):
    """Every count of columns per thread.  Along a chain of N FMAs whose terms
    change sign at random the partial sums grow like sqrt(k): RMS error 0.15 2^-24
    sum|K| whatever N, ten times that allowed; the sines (2^-23) enter as
    independent errors of the terms, 2^-24 sum|K| / sqrt(N), six times that.
    (Operands rounded to BF16 or TF32 would err by 2^-8 or 2^-11 of that.)"""
    ensure_built()
    w = inputs.kuramoto_general(n_osc=N, replicas=R, seed=N)
    ens = sde.Ensemble.kuramoto(sde.SDE_KURAMOTO_GENERAL_FP32, N, R, 0.0, 0.02, 0.005, 1)
    assert ens.tuning()[1] == 8 * tn
    K = torch.from_numpy(w["Kmat"]).cuda()
    ens.set_coupling(K)
    phi = torch.from_numpy(w["phi0"]).cuda()
    got = ens.coupling(phi).double()
    x, Kt = phi.double(), K.double().t()
    s, c = torch.sin(x), torch.cos(x)
    err = ((got - (c * (s @ Kt) - s * (c @ Kt))).abs() / K.double().abs().sum(1)).max().item() * 2 ** 24
    print("N=%d R=%d: %.2f x 2^-24 sum|K|, bound %.2f" % (N, R, err, 1.5 + 6 / math.sqrt(N)))
    assert err <= 1.5 + 6 / math.sqrt(N)


def test_members_train_in_uneven_groups():
    """Three members whose batches fill the activation rows two at a time: the
    last group is one member (the comparison of
    test_members_train_together_as_alone)."""
    test_members_train_together_as_alone(256, 2, 5, 16000, 16000)
