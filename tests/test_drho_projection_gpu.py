"""The induced density at the edges of its integer valence projection (31 terms per accumulator,
64 valence states at most) and of its weights (they go into the fields' scales), against the oracle.
Bar 1e-12 relative, that of the other FP64 density tests (the oracle's direct sums)."""
import numpy as np
import pytest

from oracle import drho as odr
from paper_2412_01695_gb300 import synth

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def density(nocc, weights, scale=1.0, spoil=None):
    torch = torch_cuda()
    from paper_2412_01695_gb300 import pwk
    pk = synth.make_config(4, k_subset=[0, 7], nb=nocc)
    pq = synth.make_config(4, k_subset=[0, 7], nb=nocc, shift_q=True)
    r = np.random.default_rng(nocc)
    du = np.zeros_like(pq.psi)
    for k in range(pq.nk):
        n = pq.npw[k]
        du[k, :, :n] = scale * (r.standard_normal((nocc, n)) + 1j * r.standard_normal((nocc, n)))
        du[k, :, :n] += 3 * scale * pq.psi[k, ::-1, :n]   # a valence part to remove
    if spoil is not None:
        du[1, 0, 3] = spoil
    plan_k, plan_q = pwk.plan_from_problem(pk), pwk.plan_from_problem(pq)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    out = torch.empty((pk.N,) * 3, dtype=torch.complex128, device="cuda")
    pwk.drho_batched(plan_q, plan_k, pwk.PWK_FP64, t(pk.psi), t(pq.psi), t(du), nocc, t(weights), out)
    torch.cuda.synchronize()
    plan_k.close()
    plan_q.close()
    return out.cpu().numpy(), (pk, pq, du)


@pytest.mark.parametrize("nocc", [1, 31, 32, 63, 64])
@pytest.mark.parametrize("weights", [(0.5, 0.5), (0.0, 1.0), (-0.3, 1e-5)])
def test_projection_and_weights(nocc, weights):
    w = np.array(weights)
    got, (pk, pq, du) = density(nocc, w)
    ref = odr.drho(pk, pq, pk.psi, pq.psi, du, weights=w)
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("exponent", [-1000, 900])
def test_fields_of_extreme_magnitude(exponent):
    s = 2.0 ** exponent
    w = np.array([0.5, 0.5])
    got, _ = density(3, w, scale=s)
    ref, _ = density(3, w)
    assert np.linalg.norm(got / s - ref) <= 1e-12 * np.linalg.norm(ref)


def test_a_non_finite_field_gives_nan():
    got, _ = density(2, np.array([0.5, 0.5]), spoil=np.inf)
    assert np.all(np.isnan(got.real))
