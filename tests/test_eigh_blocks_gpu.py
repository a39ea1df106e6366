"""pwk_eigh_batched at the edges of its blocks (16 rows per block of the triangular solves, 32
rows per warp of the Householder correction) and on either side of its two rules on threads (n =
40, 304 problems), against the oracle's reduced-problem routine; every second problem carries a
dependent basis vector, which the look-ahead factorisation drops at a block edge.

Tolerances are those of the random-pair test of the same entry point: 1e-11 of the spectrum
(backward error of a condition-1e3 pencil in FP64, 1e3 * 1e-16 * n with a margin of ten)."""
import numpy as np
import pytest

from oracle import davidson as dav

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 15, 16, 17, 31, 32, 33, 40, 41, 63, 65, 79, 81, 128, 159])
@pytest.mark.parametrize("nprob", [2, 305])
def test_block_edges(n, nprob):
    torch = torch_cuda()
    from paper_2412_01695_gb300 import pwk
    if nprob == 305 and n > 65:
        pytest.skip("the oracle's loop over 305 problems is kept short")
    rng = np.random.default_rng(100 * n + nprob)
    nev = max(1, n // 4)
    B = rng.standard_normal((2, n, 2 * n)) + 1j * rng.standard_normal((2, n, 2 * n))
    if n > 4:
        B[1, n - 1 - n % 3] = 0.5 * B[1, 0] - 2j * B[1, 1]   # dependent, beyond the first nev
    A = rng.standard_normal((2 * n, 2 * n)) + 1j * rng.standard_normal((2 * n, 2 * n))
    A = A + A.conj().T
    S, H = B.conj() @ np.swapaxes(B, 1, 2), B.conj() @ A @ np.swapaxes(B, 1, 2)
    reps = (nprob + 1) // 2
    Sd, Hd = (torch.from_numpy(np.ascontiguousarray(np.tile(M, (reps, 1, 1))[:nprob])).cuda() for M in (S, H))
    st = torch.full((nprob,), 99, dtype=torch.int32, device="cuda")
    eig, vec = pwk.eigh_batched(Hd, Sd, nev, status=st)
    assert np.all(st.cpu().numpy() == 0)
    eig, vec = eig.cpu().numpy(), vec.cpu().numpy()
    for p in range(2):
        w, _ = dav._reduced_eig(H[p], S[p], nev)
        scale = max(1.0, np.max(np.abs(w)))
        for q in range(p, nprob, 2):
            np.testing.assert_allclose(eig[q], w, rtol=0, atol=1e-11 * scale)
            assert np.array_equal(eig[q], eig[p]) and np.array_equal(vec[q], vec[p])
        X = vec[p]
        np.testing.assert_allclose(X.conj().T @ S[p] @ X, np.eye(nev), atol=1e-9)
        assert np.max(np.linalg.norm(H[p] @ X - S[p] @ X * eig[p][None, :], axis=0)) < 1e-9 * scale * np.linalg.norm(S[p], 2) ** 0.5


@pytest.mark.parametrize("n,nev", [(3, 2), (33, 8), (41, 5), (80, 20), (80, 40), (128, 32), (159, 40)])
def test_bits_do_not_depend_on_the_batch(n, nev):
    """A pencil alone, in a batch of 2 and in one of 305 (another number of threads per problem)
    gives the same bits, with and without a dependent basis vector."""
    torch = torch_cuda()
    from paper_2412_01695_gb300 import pwk
    rng = np.random.default_rng(n)
    B = rng.standard_normal((2, n, 2 * n)) + 1j * rng.standard_normal((2, n, 2 * n))
    if n > 4:
        B[1, n - 2] = 0.5 * B[1, 0] - 2j * B[1, 1]
    A = rng.standard_normal((2 * n, 2 * n)) + 1j * rng.standard_normal((2 * n, 2 * n))
    H, S = B.conj() @ (A + A.conj().T) @ np.swapaxes(B, 1, 2), B.conj() @ np.swapaxes(B, 1, 2)
    Hd, Sd = torch.from_numpy(H).cuda(), torch.from_numpy(S).cuda()
    ref = None
    for nprob in (2, 305):
        reps = (nprob + 1) // 2
        eig, vec = pwk.eigh_batched(Hd.repeat(reps, 1, 1)[:nprob].contiguous(),
                                    Sd.repeat(reps, 1, 1)[:nprob].contiguous(), nev)
        if ref is None:
            ref = eig, vec
        for p in range(2):
            assert bool((eig[p::2] == ref[0][p]).all()) and bool((vec[p::2] == ref[1][p]).all()), (nprob, p)
    for p in range(2):
        eig, vec = pwk.eigh_batched(Hd[p:p + 1].contiguous(), Sd[p:p + 1].contiguous(), nev)
        assert torch.equal(eig[0], ref[0][p]) and torch.equal(vec[0], ref[1][p])
