"""Per-particle mass matrices on the GPU (sharpy_local_metric, Sec. 5) against the
oracle's literal Fisher information on the same event arrays."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_02336_gb300 import api, inputs
from tests import gpu_helpers as G
from tests import helpers

pytestmark = pytest.mark.gpu


def _scaled_err(a, b):
    """max |a - b| / sqrt(b_jj b_kk) per particle (entries span many decades in physical units)."""
    d = np.sqrt(np.abs(np.einsum("nii->ni", b)))
    return np.max(np.abs(a - b) / (d[:, :, None] * d[:, None, :]), axis=(1, 2))


@pytest.mark.parametrize("name", ["tiny", "bbh11"])
@pytest.mark.parametrize("beta", [0.0, 0.37, 1.0])
def test_local_metric_matches_oracle(name, beta):
    G.require_gpu()
    w = inputs.WORKLOADS[name]()
    ev, ctx, th_inj, data = G.event_pair(w, seed=0)
    model = helpers.oracle_model(w)
    th = np.concatenate([inputs.prior_draws(w, 24, 5), inputs.ball(w, th_inj, 24, 6, rel=1e-3)])
    ref = oracle.local_metric(model, ev, th, beta)
    out = ctx.local_metric(G.to_dev(th), beta)
    M = out["mass"].cpu().numpy()
    assert np.max(_scaled_err(M, ref)) < 1e-8
    Mi = out["inv_mass"].cpu().numpy()
    L = out["chol"].cpu().numpy()
    eye = np.eye(w.n_dim)
    for i in range(len(th)):
        s = np.sqrt(np.diag(ref[i]))
        # M M^-1 = I in the scale of M; L L^T = M^-1; L lower triangular
        assert np.allclose((M[i] @ Mi[i]) * (1.0 / s)[:, None] * s[None, :], eye, atol=1e-6)
        assert np.allclose(L[i] @ L[i].T, Mi[i], rtol=1e-9, atol=1e-12 * np.abs(Mi[i]).max())
        assert np.allclose(np.triu(L[i], 1), 0.0)


def test_local_metric_gaussian_mixture():
    G.require_gpu()
    lo, hi = [-4.0, -2.0, -3.0], [4.0, 6.0, 3.0]
    mu, sig = [[0.5, 1.0, 0.0], [-0.5, 2.0, 1.0]], [[0.2, 0.7, 0.4], [0.3, 0.5, 0.6]]
    model = helpers.gaussmix_model(lo, hi, [0.0, -0.3], mu, sig)
    ctx = api.Context(api.gaussmix_config(lo, hi, [0.0, -0.3], mu, sig))
    th = np.random.default_rng(4).uniform(-1.0, 1.5, size=(40, 3))
    ref = oracle.local_metric(model, None, th, 0.8)
    M = ctx.local_metric(G.to_dev(th), 0.8)["mass"].cpu().numpy()
    assert np.allclose(M, ref, rtol=1e-12, atol=0)


@pytest.mark.parametrize("name", ["tiny", "bbh11"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65])
def test_local_metric_block_edges(name, n):
    """A CTA holds 32 particles: counts around its edge give, row by row, the matrices of the same particles in a
    larger call (bit for bit), each output asked for alone too, and no row past the last is written."""
    G.require_gpu()
    w = inputs.WORKLOADS[name]()
    ev, ctx, th_inj, _ = G.event_pair(w, seed=0)
    th = G.to_dev(np.concatenate([inputs.prior_draws(w, 40, 7), inputs.ball(w, th_inj, 40, 8, rel=1e-3)]))
    full = ctx.local_metric(th, 0.6)
    ref = oracle.local_metric(helpers.oracle_model(w), ev, th[:n].cpu().numpy(), 0.6)
    assert np.max(_scaled_err(full["mass"][:n].cpu().numpy(), ref)) < 1e-8
    for want in (("mass",), ("inv_mass",), ("chol",), ("mass", "inv_mass", "chol")):
        part = ctx.local_metric(th[:n].contiguous(), 0.6, want=want)
        for k in want:
            assert torch.equal(part[k], full[k][:n]), (k, want)
    guard = torch.full((n + 1, w.n_dim, w.n_dim), -7.0, dtype=torch.float64, device="cuda")
    rc = api.lib().sharpy_local_metric(ctx._h, n, api._ptr(th), 0.6, None, api._ptr(guard), None, api._stream())
    assert rc == 0 and torch.equal(guard[:n], full["inv_mass"][:n]) and bool((guard[n] == -7.0).all())


@pytest.mark.parametrize("dim", [0, 1, 2])
def test_local_metric_infinite_precision(dim):
    """A component so narrow that its precision overflows: the factorisation fails, the diagonal stays, and that
    dimension's inverse mass is 0 without touching the others."""
    G.require_gpu()
    sig = [0.1, 0.2, 0.3]
    lo, hi, mu = [-1.0] * 3, [1.0] * 3, [[0.0] * 3]
    at = G.to_dev(np.zeros((33, 3)))
    want = api.Context(api.gaussmix_config(lo, hi, [0.0], mu, [sig])).local_metric(at, 1.0)
    sig[dim] = 1e-160
    got = api.Context(api.gaussmix_config(lo, hi, [0.0], mu, [sig])).local_metric(at, 1.0)
    for k in ("inv_mass", "chol"):
        ref = want[k].clone()
        ref[:, dim, :] = 0.0
        ref[:, :, dim] = 0.0
        assert torch.allclose(got[k], ref, rtol=1e-14, atol=0.0), k
    assert torch.isinf(got["mass"][:, dim, dim]).all()
