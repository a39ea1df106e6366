"""FP64 H|psi> runs its transforms in 64-bit fixed point scaled per vector: vectors, fields and
kernel kinds at which that arithmetic could go wrong, against direct Fourier sums in long double
(the dense oracle's own FP64 sums are ten times less accurate than what is checked here).

Bar: 5e-16 relative per band: FP64 roundoff of the kinetic table and the projector sums is 2e-16
(measured with the transforms in FP64 as well), and the transforms add less, with every vector multiplied by powers of two up to 2^900 either
way, one plane wave (the largest growth in the forward transform), components of very different
size, zero and non-finite vectors, V constant, V = 0, V large and tiny."""
import numpy as np
import pytest

from paper_2412_01695_gb300 import pwk, synth

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

A = synth.fcc_lattice(7.5)
B = synth.reciprocal_rows(A)


def problem(N, V_r=None, lset=(0, 1)):
    # the largest sphere the window kernel takes on this grid
    ecut = ((N // 4 + 0.4) * 2 * np.pi / np.linalg.norm(A[0])) ** 2 * 0.9
    k = synth.mp_grid(B, (1, 1, 1)) + 0.05
    return synth.build_problem(A, np.zeros((1, 3)), lset, N, ecut, k, 4, 1, V_r=V_r, with_psi=False)


def vectors(prob):
    """Per k: normal components, one plane wave, components from 1 to 1e-12, zero."""
    r = np.random.default_rng(5)
    x = np.zeros((prob.nk, 4, prob.npw_max), complex)
    for k in range(prob.nk):
        n = prob.npw[k]
        x[k, 0, :n] = r.standard_normal(n) + 1j * r.standard_normal(n)
        x[k, 1, n // 2] = 1 - 2j
        x[k, 2, :n] = (r.standard_normal(n) + 1j * r.standard_normal(n)) * np.logspace(0, -12, n)
    return x


def apply(prob, x, shape=None, path=0):
    torch = torch_cuda()
    from paper_2412_01695_gb300 import pwk
    plan = pwk.plan_from_problem(prob)
    if shape is not None:
        plan.set_launch_shape(pwk.PWK_FP64, *shape)
    plan.set_projector_path(path)
    d = torch.from_numpy(x).cuda()
    y = torch.full_like(d, complex(np.nan, np.nan))
    pwk.hpsi_batched(plan, pwk.PWK_FP64, d, y, x.shape[1])
    torch.cuda.synchronize()
    plan.close()
    return y.cpu().numpy()


def reference(prob, k, x):
    """H x of k-point k by direct separable sums, x [nb][npw], in long double."""
    ld, cl = np.longdouble, np.clongdouble
    N, n = prob.N, int(prob.npw[k])
    pi = ld("3.14159265358979323846264338327950288")
    i = np.arange(N)
    E = np.exp(cl(2j) * pi * ((np.outer(i, i) % N).astype(ld)) / N)
    m = prob.miller[k][:n] % N
    q = prob.kpts[k][None, :] + prob.miller[k][:n] @ prob.B
    b = prob.beta[k][:, :n].astype(cl)
    out = []
    for v in x[:, :n].astype(cl):
        g = np.zeros((N, N, N), cl)
        g[m[:, 0], m[:, 1], m[:, 2]] = v
        for F, f in ((E, prob.V_r.astype(ld)), (E.conj(), ld(1) / N ** 3)):
            g = np.einsum("ai,ijk->ajk", F, g)
            g = np.einsum("bj,ajk->abk", F, g)
            g = np.einsum("ck,abk->abc", F, g) * f
        out.append(g[m[:, 0], m[:, 1], m[:, 2]] + np.sum(q * q, axis=1) * v + ((v @ b.conj().T) @ prob.D) @ b)
    return np.array(out)


def check(prob, x, y, scale=1.0):
    for k in range(prob.nk):
        n = prob.npw[k]
        ref = reference(prob, k, x[k])
        assert np.all(y[k][:, n:] == 0)
        for b in range(x.shape[1]):
            err = np.linalg.norm((y[k, b, :n] / scale - ref[b]).astype(complex))
            bar = 5e-16 * max(np.linalg.norm(ref[b].astype(complex)), np.linalg.norm(x[k, b]))
            assert err <= bar, (k, b, 5e-16 * err / max(bar, 1e-300))


@pytest.mark.parametrize("N", [12, 15, 20, 24, 25, 27, 32])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_every_kind_at_every_radix(N, kind):
    prob = problem(N)
    x = vectors(prob)
    check(prob, x, apply(prob, x, (kind, 128, 1 if kind == 2 else max(1, N // 8))))


@pytest.mark.parametrize("N", [12, 15, 32])
def test_warps_without_planes(N):
    """Kind 2 with more warps than the grid has chunks (N = 12, two planes per warp: six of eight
    warps), with a chunk each, and with several: every warp meets the same block barriers, and
    the bits are those of the CTA-wide kind."""
    prob = problem(N)
    x = vectors(prob)
    first = apply(prob, x, (1, 128, max(1, N // 4)))
    check(prob, x, first)
    for threads in (96, 128, 192, 256):
        for L in (1, 2):
            try:
                y = apply(prob, x, (2, threads, L))
            except pwk.PwkError as e:
                assert e.code == -2   # the planes of so many warps do not fit in shared memory
                continue
            assert np.array_equal(y, first), (threads, L)


@pytest.mark.parametrize("exponent", [-1060, -900, -300, 300, 900])
def test_vectors_of_any_magnitude(exponent):
    prob = problem(16)
    x = vectors(prob)
    x[:, 2] = 0   # its range would leave the doubles
    # 2^exponent in two exact steps; below 2^-1022 the inputs themselves lose bits
    half = 2.0 ** (exponent // 2)
    s = x * half * 2.0 ** (exponent - exponent // 2)
    y = apply(prob, s)
    if exponent == -1060:
        assert np.all(np.isfinite(y)) and np.any(y != 0)
        return
    check(prob, x, y / half, 2.0 ** (exponent - exponent // 2))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("path", [2, 3])
def test_a_non_finite_vector_spoils_only_itself(bad, path):
    prob = problem(16)
    x = vectors(prob)
    x[0, 2, 5] = bad
    y = apply(prob, x, path=path)
    assert np.all(~np.isfinite(y[0, 2, :prob.npw[0]]))
    y[0, 2] = 0
    x[0, 2] = 0
    check(prob, x, y)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("path,kind", [(2, 1), (3, 0), (3, 1), (3, 2)])
def test_s_of_a_non_finite_vector(bad, path, kind):
    """One component that is not finite makes every projection NaN, so all of H C and S C, in that
    vector alone."""
    torch = torch_cuda()
    prob = problem(16)
    x = vectors(prob)
    x[0, 2, 5] = bad
    plan = pwk.plan_from_problem(prob)
    plan.set_overlap(synth.random_q(np.random.default_rng(2), 1, (0, 1)))
    plan.set_projector_path(path)
    plan.set_launch_shape(pwk.PWK_FP64, kind, 128, 1)
    assert plan.projector_fused(pwk.PWK_FP64) == (path == 3)
    d = torch.from_numpy(x).cuda()
    h, s = torch.full_like(d, 7.0), torch.full_like(d, 7.0)
    pwk.hspsi_batched(plan, pwk.PWK_FP64, d, h, s, x.shape[1])
    torch.cuda.synchronize()
    plan.close()
    n = int(prob.npw[0])
    for out in (h.cpu().numpy()[0], s.cpu().numpy()[0]):
        assert np.all(np.isnan(out[2, :n].real) & np.isnan(out[2, :n].imag))
        assert np.all(np.isfinite(out[[0, 1, 3]]))


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("padding", [np.nan, 2.0 ** 600])
def test_padding_of_the_projectors_does_not_enter(kind, padding):
    """What lies beyond a sphere in beta takes no part in the scale of a projector: the same bits
    as with zeros there."""
    k = synth.mp_grid(B, (2, 2, 2))[:2] * np.array([[1.0], [0.3]]) + 0.05
    prob = synth.build_problem(A, np.zeros((1, 3)), (0, 1), 16, 20.0, k, 4, 1, with_psi=False)
    short = int(np.argmin(prob.npw))
    assert prob.npw[short] < prob.npw_max
    x = vectors(prob)
    ref = apply(prob, x, (kind, 128, 1), path=3)
    prob.beta[short, :, prob.npw[short]:] = padding
    assert np.array_equal(apply(prob, x, (kind, 128, 1), path=3), ref)


@pytest.mark.parametrize("field", ["zero", "constant", "large", "tiny", "spike", "nan"])
def test_fields(field):
    N = 20
    r = np.random.default_rng(3)
    V = {"zero": np.zeros((N,) * 3), "constant": np.full((N,) * 3, -0.75), "large": 2.0 ** 40 * r.standard_normal((N,) * 3),
         "tiny": 2.0 ** -80 * r.standard_normal((N,) * 3), "spike": np.zeros((N,) * 3),
         "nan": r.standard_normal((N,) * 3)}[field]
    if field == "spike":
        V[3, 4, 5] = -1e3
    if field == "nan":
        V[0, 0, 1] = np.nan
    prob = problem(N, V_r=V, lset=(0,))
    x = vectors(prob)
    y = apply(prob, x)
    if field == "nan":
        for k in range(prob.nk):
            assert np.all(np.isnan(y[k, :, :prob.npw[k]].real))
        return
    check(prob, x, y)


SC = synth.sc_lattice(7.5)
SITES = 7.5 * np.array([[0, 0, 0], [0, 0.5, 0.5], [0.5, 0, 0.5], [0.5, 0.5, 0]])


@pytest.mark.parametrize("N,nat,lset", [(12, 1, (0,)), (16, 4, (0, 1, 2)), (15, 1, (0, 1)), (32, 1, (0, 1)),
                                        (20, 2, (0, 1, 2))])
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("spread", [0, 150])
def test_projector_terms_in_limbs(N, nat, lset, kind, spread):
    """The projector sums inside the FP64 kernel, on the integer pipe (H alone) and in doubles (H
    and S with q): one projector, more than the 31 an accumulator holds in the add-back (36), more
    plane waves than it holds in a lane (1500 > 31 * 32), and projectors of very different size
    (2^-spread to 2^spread, the coefficients scaled back).  H and S against long double; the bar is
    that of the H tests (the limbs hold 57 bits of the largest component, the left-out products
    2^-56 of the largest product)."""
    torch = torch_cuda()
    from paper_2412_01695_gb300 import pwk
    ecut = ((N // 4 + 0.4) * 2 * np.pi / 7.5) ** 2 * 0.9
    k = synth.mp_grid(synth.reciprocal_rows(SC), (1, 1, 1)) + 0.05
    prob = synth.build_problem(SC, SITES[:nat], lset, N, ecut, k, 4, 1, with_psi=False)
    q = synth.random_q(np.random.default_rng(2), nat, lset)
    s = 2.0 ** np.linspace(-spread, spread, prob.nkb).round() if prob.nkb > 1 else np.ones(1)
    prob.beta = np.ascontiguousarray(prob.beta * s[None, :, None])
    prob.D = prob.D / np.outer(s, s)
    q = q / np.outer(s, s)
    x = vectors(prob)
    plan = pwk.plan_from_problem(prob)
    plan.set_overlap(q)
    plan.set_launch_shape(pwk.PWK_FP64, kind, 128, max(1, N // 8))
    plan.set_projector_path(3)
    assert plan.projector_fused(pwk.PWK_FP64)
    d = torch.from_numpy(x).cuda()
    h, sp = torch.full_like(d, complex(np.nan, np.nan)), torch.full_like(d, complex(np.nan, np.nan))
    pwk.hspsi_batched(plan, pwk.PWK_FP64, d, h, sp, x.shape[1])
    alone = torch.full_like(d, complex(np.nan, np.nan))
    pwk.hpsi_batched(plan, pwk.PWK_FP64, d, alone, x.shape[1])
    torch.cuda.synchronize()
    plan.close()
    check(prob, x, h.cpu().numpy())
    check(prob, x, alone.cpu().numpy())
    n = int(prob.npw[0])
    b = prob.beta[0][:, :n].astype(np.clongdouble)
    for v, got in zip(x[0], sp.cpu().numpy()[0]):
        ref = v[:n] + ((v[:n].astype(np.clongdouble) @ b.conj().T) @ q) @ b
        assert np.linalg.norm((got[:n] - ref).astype(complex)) <= 5e-16 * max(np.linalg.norm(ref.astype(complex)), 1e-300)


@pytest.mark.parametrize("path,kind", [(2, 1), (3, 0), (3, 1), (3, 2)])
@pytest.mark.parametrize("field,strength", [(0.0, 1.0), (1e-6, 1.0), (1.0, 1e4)])
def test_h_in_every_component_where_the_projectors_lead(path, kind, field, strength):
    """H C of vectors that fall off like the projectors, V = 0 or weak beside them: every
    component to the rounding of sums in doubles and of the local term.  Bound: that of S below,
    with the kinetic term (its table to four roundings), and 1e-15 max |V| |C| for the local one."""
    N, lset = 24, (0, 1)
    base = problem(N, lset=lset)
    prob = problem(N, V_r=field * base.V_r, lset=lset)
    prob.beta = strength * prob.beta
    r = np.random.default_rng(7)
    n = int(prob.npw[0])
    g = prob.kpts[0][None, :] + prob.miller[0][:n] @ prob.B
    t = np.sum(g * g, axis=1)
    x = np.zeros((1, 4, prob.npw_max), complex)
    x[0, :, :n] = np.exp(-t / 3) * (r.standard_normal((4, n)) + 1j * r.standard_normal((4, n)))
    y = apply(prob, x, (kind, 128, 1), path=path)[0, :, :n]
    b, v = np.abs(prob.beta[0][:, :n]), np.abs(x[0, :, :n])
    moduli = ((v @ b.T) @ np.abs(prob.D)) @ b
    bound = 2.0 ** -53 * 2 * ((n / 32 + 5 + 2 * prob.nkb + 4) * moduli + 4 * t * v)
    bound += 1e-15 * np.max(np.abs(prob.V_r)) * np.linalg.norm(v, axis=1)[:, None]
    assert np.all(np.abs(y - reference(prob, 0, x[0])) <= bound)


@pytest.mark.parametrize("path,kind", [(2, 1), (3, 0), (3, 1), (3, 2)])
def test_s_in_every_component(path, kind):
    """S C of vectors that fall off like the projectors (smallest components 1e-6 of the largest):
    every component to the rounding of sums in doubles, whatever its size.  Bound: u times the
    sum of moduli times the additions a term goes through (n / 32 in a lane of the projection and
    5 across lanes, nkb for delta, nkb for the add-back, two per complex product)."""
    torch = torch_cuda()
    N, lset = 24, (0, 1)
    prob = problem(N, lset=lset)
    q = synth.random_q(np.random.default_rng(2), 1, lset)
    r = np.random.default_rng(7)
    x = np.zeros((prob.nk, 4, prob.npw_max), complex)
    for k in range(prob.nk):
        n = int(prob.npw[k])
        g = prob.kpts[k][None, :] + prob.miller[k][:n] @ prob.B
        x[k, :, :n] = np.exp(-np.sum(g * g, axis=1) / 3) * (r.standard_normal((4, n)) + 1j * r.standard_normal((4, n)))
    plan = pwk.plan_from_problem(prob)
    plan.set_overlap(q)
    plan.set_projector_path(path)
    plan.set_launch_shape(pwk.PWK_FP64, kind, 128, 1)
    assert plan.projector_fused(pwk.PWK_FP64) == (path == 3)
    d = torch.from_numpy(x).cuda()
    h, s = torch.full_like(d, 7.0), torch.full_like(d, 7.0)
    pwk.hspsi_batched(plan, pwk.PWK_FP64, d, h, s, x.shape[1])
    torch.cuda.synchronize()
    plan.close()
    for k in range(prob.nk):
        n = int(prob.npw[k])
        assert np.abs(x[k, :, :n]).min() < 1e-5 * np.abs(x[k]).max()
        b, v = prob.beta[k][:, :n].astype(np.clongdouble), x[k, :, :n].astype(np.clongdouble)
        ref = v + ((v @ b.conj().T) @ q) @ b
        moduli = np.abs(v) + ((np.abs(v) @ np.abs(b).T) @ np.abs(q)) @ np.abs(b)
        bound = 2.0 ** -53 * 2 * (n / 32 + 5 + 2 * prob.nkb + 4) * moduli
        assert np.all(np.abs(s.cpu().numpy()[k, :, :n] - ref) <= bound)
