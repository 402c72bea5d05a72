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
