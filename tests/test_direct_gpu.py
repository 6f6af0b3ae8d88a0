"""GPU tests of the fixed-point predictor of Biot's system and of the face corrector, beyond the oracle parity tests:
scale invariance to the last bit, the widest ranges, and the corrector's two ways to the volume term."""
import numpy as np
import pytest

from _oracle_cases import oracle_predictor, population, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_10565_gb300 import _lib

    return _lib


def _predict(L, d, precision, q0, sweeps=1):
    ctx = L.poro_create(0, d["N"], precision)
    try:
        if precision:
            L.poro_set_refinement(ctx, sweeps)
        L.poro_set_isolated(ctx, d["vertices"], d["materials"], d["dt"])
        L.poro_set_dofs(ctx, q0)
        L.poro_predict(ctx)
        return L.poro_get_predictor(ctx, 0, q0.shape[0])
    finally:
        L.poro_destroy(ctx)


@pytest.mark.parametrize("precision,sweeps,powers", [(0, 1, (-900, -300, 300, 900)), (1, 1, (-60, 60)), (1, 2, (-300, 300))])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
def test_power_of_two_scaling_is_exact(L, N, precision, sweeps, powers):
    """The fixed-point scales are powers of two that follow the data, so Q0 times 2^k gives the predictor times 2^k bit by
    bit (away from the ends of the arithmetic's range: the star products carry up to about 1e+-20)."""
    d = population(7, N, seed=800 + N)
    ref = _predict(L, d, precision, d["Q0"], sweeps)
    for k in powers:
        got = _predict(L, d, precision, np.ldexp(d["Q0"], k), sweeps)
        np.testing.assert_array_equal(np.ldexp(got, -k), ref, err_msg=f"2^{k}")


@pytest.mark.parametrize("N", [1, 3, 6])
def test_smallest_binary64_data(L, N):
    """Velocities near the lower end of binary64's range: the stresses and pressure that follow from them (2^20 times as
    large, so that nothing on the way leaves the normal range) are as accurate as those of data of ordinary size."""
    d = population(5, N, seed=850 + N)
    q0 = d["Q0"].copy()
    q0[:, :6] = q0[:, 9] = 0.0
    ref, got = _predict(L, d, 0, q0), _predict(L, d, 0, np.ldexp(q0, -1010))
    for p in (0, 1, 2, 3, 4, 5, 9):
        assert rel_l2(np.ldexp(got[:, p], 1010), ref[:, p]) <= 1e-14, p


@pytest.mark.parametrize("N", [1, 3, 6])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-10), (2, 1e-10)])
def test_rows_of_unlike_size(L, N, precision, tol):
    """Quantities many orders of magnitude apart (stresses in Pa beside velocities in m/s), zero rows among them: every
    quantity of the predictor is accurate by itself where the data reach it at its own size."""
    d = population(5, N, seed=900 + N)
    q0 = d["Q0"].copy()
    q0[:, [0, 1, 2, 3, 4, 5, 9]] *= 1e7
    q0[:, 10:] = 0.0
    q0[1] = 0.0
    qt = _predict(L, d, precision, q0)
    assert not qt[1].any()
    d = dict(d, Q0=q0)
    for i in (0, 2, 3, 4):
        ref = oracle_predictor(d, i)
        for p in range(13):
            assert rel_l2(qt[i, p], ref[p]) <= tol, (i, p)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("mode", [0, -1])
def test_non_finite_binary64_rows(L, bad, mode):
    """A non-finite entry of one element's data makes what depends on it non-finite and touches no other element."""
    N = 4
    d = population(6, N, seed=77)
    q0 = d["Q0"].copy()
    q0[2, 7, mode] = bad
    clean, dirty = _predict(L, d, 0, d["Q0"]), _predict(L, d, 0, q0)
    keep = np.arange(6) != 2
    np.testing.assert_array_equal(clean[keep], dirty[keep])
    assert not np.isfinite(dirty[2, 7]).all()
    if mode == -1:  # the last mode feeds the lower ones
        assert not np.isfinite(dirty[2, :, 0]).all()


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("precision,sweeps,tol", [(0, 1, 1e-13), (1, 1, 1e-11), (2, 2, 1e-11), (1, 0, 1e-4), (2, 0, 1e-2)])
def test_step_equals_predict_and_correct(L, N, precision, sweeps, tol):
    """One time step of poro_advance (the predictor writes Q~(1), the corrector adds the faces) against poro_predict and
    poro_correct (volume term from the time integral, then the faces); with no refinement sweep both take the second
    way, and the step is compared with binary64's.  Free surface, absorbing and interior faces of two materials."""
    from paper_2108_10565_gb300 import inputs

    mesh = inputs.kuhn_box_mesh((3, 2, 2), lo=(0, 0, -1), hi=(1.5, 1.2, 0), periodic=(True, False, False), tags={"z+": 1})
    ne = mesh["tets"].shape[0]
    z = mesh["vertices"][mesh["tets"]].mean(axis=1)[:, 2]
    mats = np.where((z > -0.5)[:, None], inputs.REFERENCE_MATERIAL, inputs.HALFSPACE_MATERIAL)
    q0 = np.random.default_rng(N).standard_normal((ne, 13, (N + 1) * (N + 2) * (N + 3) // 6))

    def run(prec, advance):
        ctx = L.poro_create(0, N, prec)
        try:
            if prec:
                L.poro_set_refinement(ctx, sweeps)
            L.poro_set_mesh(ctx, mesh["vertices"], mesh["tets"], mesh["neighbors"], mesh["face_tag"])
            L.poro_set_materials(ctx, mats)
            dt, _ = L.poro_set_clusters(ctx, 0.5, 1)
            L.poro_set_dofs(ctx, q0)
            if advance:
                L.poro_advance(ctx, 1.5 * dt)
            else:
                L.poro_predict(ctx)
                L.poro_correct(ctx)
            return L.poro_get_dofs(ctx)
        finally:
            L.poro_destroy(ctx)

    a, b = run(precision, True), run(precision if sweeps else 0, False)
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("precision", [0, 1])
def test_launch_sizes_agree(L, N, precision):
    """The CTA size that a launch takes by its number of elements (one, two or four CTAs an SM, or more) does not change
    a bit of the predictor."""
    d = population(613, N, seed=700 + N)
    ctx = L.poro_create(0, N, precision)
    try:
        L.poro_set_isolated(ctx, d["vertices"], d["materials"], d["dt"])
        L.poro_set_dofs(ctx, d["Q0"])
        L.poro_set_variant(ctx, 1)
        L.poro_predict(ctx)
        ref = L.poro_get_predictor(ctx, 0, 613)
    finally:
        L.poro_destroy(ctx)
    for n in (1, 152, 153, 304, 305, 608, 609):
        part = {k: d[k][:n] for k in ("vertices", "materials")}
        got = _predict(L, dict(part, N=N, dt=d["dt"]), precision, d["Q0"][:n])
        np.testing.assert_array_equal(got, ref[:n], err_msg=f"{n} elements")


def _advance(L, N, precision, mesh, q0, steps, sweeps=1):
    from paper_2108_10565_gb300 import inputs

    ctx = L.poro_create(0, N, precision)
    try:
        if precision:
            L.poro_set_refinement(ctx, sweeps)
        L.poro_set_mesh(ctx, mesh["vertices"], mesh["tets"], mesh["neighbors"], mesh["face_tag"])
        L.poro_set_materials(ctx, np.tile(inputs.REFERENCE_MATERIAL, (mesh["tets"].shape[0], 1)))
        dt, _ = L.poro_set_clusters(ctx, 0.5, 1)
        L.poro_set_dofs(ctx, q0)
        L.poro_advance(ctx, (steps + 0.5) * dt)
        return L.poro_get_dofs(ctx)
    finally:
        L.poro_destroy(ctx)


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("precision", [1, 2])
def test_mixed_steps_carry_the_field_in_binary64(L, N, precision):
    """The double-binary32 predictor gives a step's change, and the field itself stays in binary64.  A uniform field
    without relative fluid flow does not change (the two sides of every face are equal word by word, so the change is
    zero), and entries below binary32's range (whose change is then zero) stay as they are."""
    from paper_2108_10565_gb300 import inputs

    mesh = inputs.kuhn_box_mesh(3)
    ne, B = mesh["tets"].shape[0], (N + 1) * (N + 2) * (N + 3) // 6
    rng = np.random.default_rng(N)
    q0 = np.zeros((ne, 13, B))
    q0[:, :10, 0] = rng.standard_normal(10) * np.r_[np.full(6, 1e7), np.ones(3), 1e7]
    np.testing.assert_array_equal(_advance(L, N, precision, mesh, q0, 3), q0)
    q0 = rng.standard_normal((ne, 13, B)) * 1e-60
    np.testing.assert_array_equal(_advance(L, N, precision, mesh, q0, 3), q0)


@pytest.mark.parametrize("N", [2, 3])
def test_mixed_steps_do_not_drift(L, N):
    """Thousands of mixed steps against as many in binary64, elements 1e-9 of the field's size among them: every step
    rounds its change in about 2^-48, so that n steps are within n 2^-48 of the field's size."""
    from paper_2108_10565_gb300 import inputs

    steps = 4000
    mesh = inputs.kuhn_box_mesh(3)
    ne, B = mesh["tets"].shape[0], (N + 1) * (N + 2) * (N + 3) // 6
    q0 = np.random.default_rng(N).standard_normal((ne, 13, B)) * np.r_[np.full(6, 1e7), np.ones(3), 1e7, np.zeros(3)][:, None]
    q0[::2] *= 1e-9
    a, b = _advance(L, N, 1, mesh, q0, steps), _advance(L, N, 0, mesh, q0, steps)
    for p in range(13):
        err = np.abs(a[:, p] - b[:, p]).max() / np.abs(b[:, p]).max()
        assert err <= steps * 2.0 ** -48, (p, err)


def _autotune(L, N, n, sample, precision=0):
    d = population(n, N, seed=600 + N)
    ctx = L.poro_create(0, N, precision)
    try:
        L.poro_set_isolated(ctx, d["vertices"], d["materials"], d["dt"])
        L.poro_set_dofs(ctx, d["Q0"])
        L.poro_predict(ctx)
        before = L.poro_get_predictor(ctx, 0, n)
        best, ms = L.poro_autotune(ctx, sample)
        tile, tile_ms = L.poro_autotune_tiles(ctx, sample)
        L.poro_predict(ctx)
        np.testing.assert_array_equal(L.poro_get_predictor(ctx, 0, n), before)
        return best, list(ms), tile, list(tile_ms)
    finally:
        L.poro_destroy(ctx)


@pytest.mark.parametrize("N", [1, 3])
def test_autotuners_time_one_kernel_once(L, N):
    """Up to 4 elements an SM both variants are the same kernel at N <= 3 (128 threads; at N = 3 up to two an SM 256): the
    tuners time it once and keep variant 0."""
    for n in (100, 400):
        best, ms, tile, tile_ms = _autotune(L, N, n, 0)
        assert best == 0 and ms[0] == ms[1] > 0
        assert tile == 0 and tile_ms[0] == tile_ms[6] > 0


def test_autotuners_time_the_kernel_that_runs(L):
    """A sample of 100 elements out of 2,000 would be launched with a CTA size that 2,000 are not: the tuners time as many
    as take the population's size (over 4 an SM, here at 3 CTAs an SM: two waves and more, against one)."""
    _, small, _, small_tiles = _autotune(L, 5, 100, 0)
    _, ms, _, tile_ms = _autotune(L, 5, 2000, 100)
    assert ms[0] > 1.5 * small[0] and tile_ms[0] > 1.5 * small_tiles[0]
