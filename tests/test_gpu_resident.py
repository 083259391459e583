"""Small-mesh solves as one resident launch (csrc/resident.cu) against the
oracle, at the sizes where its layout changes: one CTA or a cluster of 2, 4, 8
or (Jacobi) 16 per sample, bands with an odd last slab, levels split or on one
CTA, the largest meshes it takes and the first ones it leaves to the separate
kernels (3D multigrid: 32^3, in test_gpu_parity3d.py).

Tolerances: the solve stops at ||r|| <= 1e-11 ||b||, so Q is within 1e-9 and u
within 1e-7 of the oracle's direct solution (the bounds of the other solves)."""
import functools
from fractions import Fraction

import numpy as np
import pytest

from oracle import fem, mlmc as omlmc
from synth import random_element_field, small_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_11788_gb300.build import build_library
    build_library()
    import paper_2111_11788_gb300.mlmc as mod
    mod.lib()
    return mod


def stream():
    return torch.cuda.current_stream().cuda_stream


def solve(m, dim, n, solver, precision, kap, **over):
    count, ne, nn = kap.shape[0], n ** dim, (n + 1) ** dim
    cfg = m.config(dim=dim, n_levels=1, coarse_cells=n, solver=solver, rtol=1e-11, precision=precision, **over)
    es, ns = m.elem_stride(dim, n), m.node_stride(dim, n)
    k = torch.zeros(count, es, dtype=torch.float64)
    k[:, :ne] = torch.from_numpy(kap)
    k = k.cuda()
    u = torch.full((count, ns), float("nan"), dtype=torch.float64, device="cuda")
    q = torch.zeros(count, dtype=torch.float64, device="cuda")
    it = torch.zeros(count, dtype=torch.int32, device="cuda")
    with m.Plan(cfg, stream()) as plan:
        st = plan.solve(0, k.data_ptr(), count, u.data_ptr(), q.data_ptr(), it.data_ptr(), allow_not_converged=True)
    return st, u.cpu().numpy()[:, :nn], q.cpu().numpy(), it.cpu().numpy()


SIZES = [(2, "gmg", n) for n in (2, 4, 8, 16, 32, 64, 128, 256)] + \
        [(2, "jacobi", n) for n in (2, 3, 23, 33, 45, 67, 100, 131, 170, 171, 256, 257)] + \
        [(3, "gmg", n) for n in (4, 8, 16)] + [(3, "jacobi", n) for n in (3, 9, 13, 18, 24, 25, 30, 31)]


@functools.lru_cache(maxsize=None)
def reference(dim, n):
    """Element coefficients and the oracle's solutions (the larger 3D meshes, slow there: one sample)."""
    kap = random_element_field(dim, n, 2 if n ** dim < 20 ** 3 or dim == 2 else 1, seed=11 * n + dim, spread=0.7)
    b = fem.load_vector(dim, n)
    return kap, [fem.solve(fem.assemble_fast(dim, n, k), b, dim) for k in kap]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,solver,n", SIZES)
def test_solve_matches_oracle(m, dim, solver, n, precision):
    kap, refs = reference(dim, n)
    qoi = "box" if n % 4 == 0 else "domain"
    st, u, q, it = solve(m, dim, n, solver, precision, kap, qoi=qoi)
    assert st == 0 and np.all(it > 0)
    w = fem.qoi_weights(dim, n, qoi)
    for s, ref in enumerate(refs):
        assert abs(q[s] - w @ ref) <= 1e-9 * abs(w @ ref)
        assert np.max(np.abs(fem.from_node_grid(dim, n, u[s]) - ref)) <= 1e-7 * np.max(np.abs(ref))
        # boundary nodes are written as 0
        full = u[s].reshape([n + 1] * dim)
        for a in range(dim):
            assert not full.take([0, n], axis=a).any()


@pytest.mark.parametrize("dim,solver,precision,last,first_left", [
    (2, "gmg", "fp64", 128, 256), (2, "gmg", "mixed", 128, 256), (3, "gmg", "fp64", 16, 32), (3, "gmg", "mixed", 16, 32),
    (2, "jacobi", "fp64", 170, 171), (2, "jacobi", "mixed", 256, 257), (3, "jacobi", "fp64", 24, 25),
    (3, "jacobi", "mixed", 30, 31)])
def test_the_meshes_that_run_resident(m, dim, solver, precision, last, first_left):
    """By the launches of a solve: two of setup and the solve, against hundreds of the separate kernels. The meshes
    beyond `last` are those where 100 samples are faster on the separate kernels."""
    for n, resident in ((last, True), (first_left, False)):
        cfg = m.config(dim=dim, n_levels=1, coarse_cells=n, solver=solver, precision=precision, rtol=1e-8)
        k = torch.ones(m.elem_stride(dim, n), dtype=torch.float64, device="cuda")
        u = torch.zeros(m.node_stride(dim, n), dtype=torch.float64, device="cuda")
        q = torch.zeros(1, dtype=torch.float64, device="cuda")
        with m.Plan(cfg, stream()) as plan:
            before = plan.launch_count()
            plan.solve(0, k.data_ptr(), 1, u.data_ptr(), q.data_ptr(), 0)
            torch.cuda.synchronize()
            assert (plan.launch_count() - before <= 3) == resident, n


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,solver,n", [(2, "gmg", 64), (2, "jacobi", 45), (3, "gmg", 16), (2, "gmg", 8),
                                          (2, "jacobi", 67), (2, "jacobi", 100), (3, "jacobi", 18), (3, "jacobi", 23)])
def test_results_do_not_depend_on_the_batch(m, dim, solver, n, precision):
    """One band per CTA alone, two or four in the batch (Jacobi from 66^2 and 18^3 on: 16 bands)."""
    kap = random_element_field(dim, n, 200, seed=5, spread=0.5)
    _, u, q, it = solve(m, dim, n, solver, precision, kap)
    for s in (0, 7, 199):
        _, u1, q1, it1 = solve(m, dim, n, solver, precision, kap[s:s + 1])
        assert np.array_equal(u1[0], u[s]) and q1[0] == q[s] and it1[0] == it[s]


@pytest.mark.parametrize("solver,n", [("gmg", 64), ("jacobi", 45)])
def test_iteration_caps(m, solver, n):
    kap = random_element_field(2, n, 3, seed=9, spread=0.5)
    st, _, _, it = solve(m, 2, n, solver, "fp64", kap, max_iter=2)
    assert st == m.MLMC_ERR_NOT_CONVERGED and np.all(it == -1)
    # mixed form: inner solves cut at one iteration each still refine (their iterations are counted); the
    # outer cap ends the solve
    st, _, _, it = solve(m, 2, n, solver, "mixed", kap, inner_max_iter=1, outer_max_iter=2)
    assert st == m.MLMC_ERR_NOT_CONVERGED and np.all(it == -1)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,solver,n0,levels", [(2, "gmg", 32, 4), (2, "jacobi", 25, 3), (3, "gmg", 4, 4)])
def test_coupled_samples_with_the_nested_guess(m, dim, solver, n0, levels, precision):
    """Pairs on both sides of the size where the resident solve ends."""
    wl = small_case(dim, n0=n0, levels=levels, m=3, solver=solver, rtol=1e-11, precision=precision)
    with m.Plan(m.config_from_workload(wl), stream()) as plan:
        for level in range(levels):
            qf, qc, it = plan.sample_level(level, 5, 2)
            assert np.all(it > 0)
            a, b = omlmc.coupled_sample(wl, level, 6)
            assert abs(qf[1] - a) <= 1e-9 * abs(a)
            assert level == 0 or abs(qc[1] - b) <= 1e-9 * abs(b)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_round_with_larger_meshes(m, precision):
    """Resident solves held to a share of the GPU, clusters taking several samples in turn: the same samples."""
    wl = small_case(2, n0=32, levels=4, m=3, solver="gmg", precision=precision, N=(400, 130, 3, 2))
    cfg = m.config_from_workload(wl)
    with m.Plan(cfg, stream()) as plan, m.Plan(cfg, stream()) as ref:
        plan.run(N=wl["N"])
        for level, count in enumerate(wl["N"]):
            qf, qc, _ = ref.sample_level(level, 0, count)
            n, mean, m2 = plan.level_stats(level)[:3]
            y = np.asarray(qf) - (np.asarray(qc) if level else 0.0)
            # Welford's update rounds a few ulps of the largest value per sample
            assert n == count and abs(mean - y.mean()) <= 4 * count * 2.0 ** -53 * np.abs(y).max()


@pytest.mark.parametrize("dim,n,precision,count", [(2, 256, "fp64", 120), (2, 256, "mixed", 120), (2, 512, "mixed", 60),
                                                   (3, 32, "fp64", 240), (3, 64, "mixed", 120)])
def test_fused_levels_do_not_depend_on_the_batch(m, dim, n, precision, count):
    """Larger meshes: the V-cycle's small levels on a cluster whose size follows the batch."""
    kap = random_element_field(dim, n, 2, seed=6, spread=0.5)
    _, u, q, it = solve(m, dim, n, "gmg", precision, np.concatenate([kap] * (count // 2)))
    assert np.all(it > 0)
    for s in (0, 1):
        _, u1, q1, it1 = solve(m, dim, n, "gmg", precision, kap[s:s + 1])
        for k in (s, count - 2 + s):
            assert np.array_equal(u1[0], u[k]) and q1[0] == q[k] and it1[0] == it[k]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,solver,n0,count", [(2, "gmg", 32, 130), (2, "jacobi", 22, 150), (3, "gmg", 8, 150),
                                                 (2, "jacobi", 50, 64), (3, "jacobi", 9, 130)])
def test_coupled_batches_repeat_bitwise(m, dim, solver, n0, count, precision):
    """CTAs of several bands: a batch gives the same bits every time, and each sample the bits of a call of its own."""
    wl = small_case(dim, n0=n0, levels=2, m=3, solver=solver, precision=precision)
    with m.Plan(m.config_from_workload(wl), stream()) as plan:
        one = [plan.sample_level(1, k, 1) for k in range(count)]
        want = [np.concatenate([np.atleast_1d(o[i]) for o in one]) for i in (0, 1)]
        for _ in range(8):
            qf, qc, _ = plan.sample_level(1, 0, count)
            assert np.array_equal(qf, want[0]) and np.array_equal(qc, want[1])


@pytest.mark.parametrize("dim", [2, 3])
def test_mixed_residual_is_rounded_once(m, dim):
    """One unknown, an FP32 operator that inverts exactly (4 in 2D, 2 in 3D) and an FP64 one off it by less than half
    an FP32 unit: the second refinement step's right-hand side r / ||r|| is then -1 in FP32, and it removes the whole
    FP64 residual of the first. The operator's entry, the residual and the solution round to 2^-53 each; a residual
    rounded to FP32 before it is scaled misses by a further 2^-24 of the correction (2e-15 of u)
    on some of the samples."""
    count, b, d = 256, 0.5 ** dim, 4.0 if dim == 2 else 2.0
    eps = 3e-8 + np.arange(count) * 3.5e-11
    kap = np.repeat(1.5 * (1.0 + eps)[:, None], 2 ** dim, axis=1)
    assert np.all(kap.astype(np.float32) == np.float32(1.5))
    st, u, _, it = solve(m, dim, 2, "jacobi", "mixed", kap, outer_max_iter=2)
    assert st == 0 and np.all(it == 2)
    D = [Fraction(d) * Fraction(k) / Fraction(3, 2) for k in kap[:, 0]]
    u1 = Fraction(b) / Fraction(d)
    want = np.array([float(u1 + (Fraction(b) - x * u1) / Fraction(d)) for x in D])
    got = u.reshape([count] + [3] * dim)[(slice(None),) + (1,) * dim]
    assert np.max(np.abs(got - want) / want) <= 5 * 2.0 ** -53
