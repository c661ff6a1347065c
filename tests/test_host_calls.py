"""Host code of the library's calls on a stand-in for the CUDA runtime (fake_runtime.py; no GPU)."""
import contextlib

import numpy as np
import pytest

import fake_runtime
import synth
from oracle import poisson
from paper_1003_4570_gb300 import omen


@pytest.fixture(scope="module")
def watch(tmp_path_factory):
    with fake_runtime.loaded(tmp_path_factory.mktemp("host")) as w:
        yield w


@pytest.fixture
def ctx(watch):
    watch.reset()
    return omen.omen_create(0)


def test_poisson_never_lowers_a_shared_memory_limit(watch, ctx):
    """The limit is the kernel's, shared by every context: a small plane or line after a large one
    must leave it, or a large solve of another thread fails between its setting and its launch."""
    for sizes in [((55, 55, 9), (43, 41, 9)), ((2048, 3, 9), (1600, 3, 9)), ((9, 2048, 9), (9, 1600, 9))]:
        for n in sizes:
            f = np.zeros((n[2] - 1, n[1], n[0]))
            omen.omen_poisson(ctx, poisson.Grid(*n, 1.0, 1.0, 1.0), f, f.copy())
    assert watch.lowered() == 0


def hamiltonian(ctx, cells, basis=10, bloch=False, precision=omen.OMEN_F64):
    lat = omen.omen_build_lattice(ctx, synth.lattice_spec(*cells, (2, 2, 0) if bloch else (0, 0, 0), seed=1))
    return omen.omen_assemble_H(ctx, lat, synth.draw_tb_params(1, basis, 1), precision=precision,
                                k=(0.1, 0.2, 0.0) if bloch else None)


@pytest.mark.parametrize("precision", [omen.OMEN_F64, omen.OMEN_F32, omen.OMEN_F64_DF])
@pytest.mark.parametrize("which", [omen.OMEN_LOWEST, omen.OMEN_NEAREST])
@pytest.mark.parametrize("bloch", [False, True])
def test_coefficients_outlive_their_copy(watch, ctx, precision, which, bloch):
    """A pending copy may read host memory until the stream is synchronised: what a solve's restarts
    and Ritz vectors copy from must be left alone until then (3 and 40 vectors: both of its routes)."""
    if bloch and precision == omen.OMEN_F64_DF:
        pytest.skip("double-float Hamiltonians are real")
    ham = hamiltonian(ctx, (2, 3, 4), bloch=bloch, precision=precision)
    for nev in (3, 40):
        omen.omen_eigs(ctx, ham, nev, which, block=1, basis=96, raise_on_noconv=False)
        assert watch.changed() == 0, nev


def test_wave_vectors_outlive_their_copy(watch, ctx):
    ham = hamiltonian(ctx, (2, 2, 3), bloch=True)
    k = np.random.default_rng(1).normal(size=(300, 3))
    x = np.zeros((300, ham.nrows), complex)
    omen.omen_hx_kbatch(ctx, ham, k, x, np.zeros_like(x))
    omen.omen_eigs_kbatch(ctx, ham, k[:5], 4, raise_on_noconv=False)
    assert watch.changed() == 0


@pytest.mark.parametrize("call", ["eigs", "refined", "kbatch", "host"])
def test_a_failed_allocation_leaves_nothing_behind(watch, ctx, call):
    prec = {"refined": omen.OMEN_F32_REFINE64, "host": omen.OMEN_F64_DF}.get(call, omen.OMEN_F64)
    ham = hamiltonian(ctx, (2, 2, 3), bloch=call == "kbatch", precision=prec)
    before, failed = watch.live(), 0
    for n in range(60):
        watch.fail(n)
        try:
            if call == "host":
                omen.omen_hx_host(ctx, ham, np.zeros(ham.nrows))
            elif call == "kbatch":
                omen.omen_eigs_kbatch(ctx, ham, np.zeros((3, 3)), 4, raise_on_noconv=False)
            else:
                omen.omen_eigs(ctx, ham, 4, block=1, basis=32, raise_on_noconv=False)
        except omen.OmenError as e:
            failed += e.status == omen.OMEN_ENOMEM
        assert watch.live() == before, n
    watch.fail(-1)
    assert failed >= (3 if call == "host" else 15)


ITERATED = [((2039, 2039, 2), 1e-13), ((1021, 1021, 5), 1e-13), ((2039, 16, 3), 1e-6), ((1, 2039, 3), 1e-10), ((2053, 1, 3), 1e-9),
            ((1, 1, 1100), 1e-9)]
DIRECT = [((1, 1, 2), 1e-13), ((11, 11, 217), 1e-13), ((16, 13, 20), 1e-13), ((251, 241, 25), 1e-10), ((24, 251, 25), 1e-10),
          ((251, 24, 25), 1e-10), ((53, 53, 9), 1e-6), ((1024, 1024, 2), 1e-13), ((251, 251, 25), 1e-6), ((2048, 2048, 2), 1e-6),
          ((256, 256, 25), 1e-3), ((509, 509, 33), 1e-13)]


@pytest.mark.parametrize("precision", [omen.OMEN_F64, omen.OMEN_F32_REFINE64])
@pytest.mark.parametrize("n, rtol", ITERATED + DIRECT)
def test_poisson_takes_the_faster_form(watch, ctx, n, rtol, precision):
    """Lines with a large prime and few planes are iterated, the rest is solved directly; a limit on
    the iterations that the iterated form might not keep leaves the direct one."""
    f = np.zeros((n[2] - 1, n[1], n[0]))
    iterated, fits = (n, rtol) in ITERATED, n[0] <= 2048 and n[2] <= 1025
    if precision == omen.OMEN_F32_REFINE64 and rtol < 1e-12:
        iterated = False
    for limit in (100000, 20):
        watch.reset()
        with contextlib.suppress(omen.OmenError):      # the stand-in's iterations do not converge
            omen.omen_poisson(ctx, poisson.Grid(*n, 0.2 * n[0], 0.2 * n[1], 0.2 * n[2]), f, f.copy(), rtol=rtol, precision=precision,
                              max_iter=limit)
        assert (watch.launches("cg_") == 1) == (iterated and (limit > 20 or not fits)), limit


# (Ritz vectors combined, passes of 8, 16 and 25 columns): whole passes without idle columns where that
# costs no extra pass
@pytest.mark.parametrize("cols, passes", [(9, (0, 1, 0)), (17, (0, 0, 1)), (32, (0, 2, 0)), (33, (1, 0, 1)), (49, (0, 0, 2)),
                                          (51, (1, 0, 2)), (64, (0, 1, 2))])
def test_passes_of_a_restart(watch, ctx, cols, passes):
    ham = hamiltonian(ctx, (2, 2, 3))
    omen.omen_set_locking_check(ctx, False)
    omen.omen_eigs(ctx, ham, cols - 1, block=1, basis=96, raise_on_noconv=False)
    assert tuple(watch.launches(f"combine_split_kernelILi{n}E") for n in (8, 16, 25)) == passes


@pytest.mark.parametrize("precision", [omen.OMEN_F64, omen.OMEN_F32])
@pytest.mark.parametrize("cells, ahead", [((2, 2, 3), True), ((16, 16, 16), True), ((24, 24, 24), False)])
def test_steps_ahead_of_a_check(watch, ctx, cells, ahead, precision):
    """Small problems queue the next segment while the host looks at the check before it; larger ones do
    not where that check may end the solve: here its first one does, and only the steps reported run."""
    ham = hamiltonian(ctx, cells, basis=5, precision=precision)
    omen.omen_set_locking_check(ctx, False)
    info = omen.omen_eigs(ctx, ham, 4, block=1, basis=48, raise_on_noconv=False)[1]
    assert info["iterations"] == 12
    assert watch.launches("update_norm_kernel") == (24 if ahead else 12)


@pytest.mark.parametrize("cells, tuned", [((2, 2, 3), False), ((10, 10, 10), False), ((20, 20, 20), True)])
def test_tuner_keeps_the_built_in_shape_of_small_products(watch, ctx, cells, tuned):
    """Small products take one kernel whatever shape is set, so the times of its launches (here each
    shorter than the one before) say nothing; of larger ones every distinct launch is timed once."""
    ham = hamiltonian(ctx, cells, precision=omen.OMEN_F32)
    r = omen.omen_tune_hx(ctx, ham, reps=1)
    assert r["candidates"] == 12                       # four widths, one, two or four bonds' loads
    if tuned:
        assert (r["threads"], r["rows_per_batch"]) == (128, 5) and r["ms_best"] < r["ms_default"]
        assert watch.launches("hx_kernel") == 3 * 12
    else:
        assert (r["threads"], r["rows_per_batch"]) == (128, 0) and r["ms_best"] == r["ms_default"]
        assert watch.launches("hx_kernel") == 0


def test_host_tables_of_asynchronous_calls_may_go(watch, ctx):
    """What a call that does not wait was given by host pointer is read when it returns."""
    ham = hamiltonian(ctx, (2, 2, 3))
    psi, n = np.zeros((70, ham.nrows)), np.zeros(96)
    occ, weight = np.ones(70), np.ones(70)
    omen.omen_density_accum(ctx, ham, psi, 70, occ, 1.0, n)
    omen.omen_state_weights(ctx, ham, psi, 70, weight, np.zeros((70, 96)))
    occ[:], weight[:] = 2.0, 3.0
    assert watch.changed() == 0
    spec = synth.lattice_spec(1, 1, 4, (2, 2, 0), seed=1)
    g = poisson.Grid(3, 3, 12, 0.5431, 0.5431, 4 * 0.5431)
    f = np.zeros(g.shape)
    omen.omen_scf(ctx, omen.omen_build_lattice(ctx, spec), synth.draw_tb_params(1, 10, 1), g, f, f.copy(), 2.0, 0.01, [[0, 0, 0]],
                  [1.0], 4, 0.0, -1.0, max_iter=4, mix_history=3, raise_on_noconv=False)
    assert watch.changed() == 0


def test_relaxation_refuses_species_outside_its_table(watch, ctx):
    """The kernels look constants up by the species of an atom: an index above 3 would leave the table."""
    class Keating:
        a_nm, alpha, beta = np.full(4, 0.5431), np.full(4, 300.0), np.full(4, 90.0)
    for bad in (3, 4, 255):
        spec = synth.lattice_spec(1, 2, 2, (0, 0, 0), seed=1)
        spec.species[5] = bad
        lat, u = omen.omen_build_lattice(ctx, spec), np.zeros((3, spec.natoms))
        calls = [lambda: omen.omen_vff_energy_forces(ctx, lat, Keating, u), lambda: omen.omen_relax_vff(ctx, lat, Keating, u, max_iter=0)]
        for call in calls:
            if bad <= 3:
                call()
            else:
                with pytest.raises(omen.OmenError, match="EINVAL"):
                    call()
