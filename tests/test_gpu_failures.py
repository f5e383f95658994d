"""Failure paths, made to happen without faulting or hanging the GPU.

* A bounded wait that runs out: the TMA producer is told to skip one source row
  (tclbm_test_skip_row); the consumers' 1 s waits expire, the kernel records the failure
  and returns, and the next synchronising call reports TCLBM_ETIMEOUT.  The context
  stays usable: the same handle, re-initialised, steps correctly afterwards.
* An allocator hook that returns NULL: tclbm_create reports TCLBM_ENOMEM.
* A non-finite state: the FP64 diagnostics report TCLBM_ENONFINITE.
"""
import ctypes

import numpy as np
import pytest

from paper_1610_07114_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1610_07114_gb300 import build

    build.build()
    from paper_1610_07114_gb300 import tclbm

    return tclbm


def test_expired_pipeline_wait_is_reported_and_the_context_recovers(T):
    case, fields = W.rayleigh_benard(256, 64, Ra=1e4, seed=9)
    ref = T.Lattice(case, fields)
    ref.set_kernel(0)
    ref.step(5)
    f_ref, h_ref = ref.populations()
    ref.close()

    lat = T.Lattice(case, fields)
    lat.set_kernel(0)
    T.tclbm_test_skip_row(lat.handle, 30)
    lat.step(1)
    with pytest.raises(T.TclbmError) as err:
        lat.diagnostics()
    assert err.value.status == T.ETIMEOUT
    T.tclbm_test_skip_row(lat.handle, -1)
    lat.init_fields(fields)
    lat.step(5)
    f, h = lat.populations()
    lat.close()
    assert np.array_equal(f, f_ref) and np.array_equal(h, h_ref)


def test_expired_wait_in_a_chain_of_launches_is_reported_and_the_context_recovers(T):
    # three chained launches: the first one's CTA for row 30 never gets that row and
    # gives up after 1 s; the items of the next launches that wait for it see the error
    # word and return instead of waiting out their own limit
    case, fields = W.rayleigh_benard(1024, 512, Ra=1e4, seed=9)
    ref = T.Lattice(case, fields)
    ref.set_kernel(0)
    ref.set_tile(128, 16)
    ref.step(5)
    f_ref, h_ref = ref.populations()
    ref.close()

    lat = T.Lattice(case, fields)
    lat.set_kernel(0)
    lat.set_tile(128, 16)
    T.tclbm_test_skip_row(lat.handle, 30)
    lat.step(3)
    with pytest.raises(T.TclbmError) as err:
        lat.diagnostics()
    assert err.value.status == T.ETIMEOUT
    T.tclbm_test_skip_row(lat.handle, -1)
    lat.init_fields(fields)
    lat.step(5)
    f, h = lat.populations()
    lat.close()
    assert np.array_equal(f, f_ref) and np.array_equal(h, h_ref)


def test_expired_wait_of_a_resident_run_is_reported_and_the_context_recovers(T):
    # row 12 is the edge of a tile that never publishes it: the tiles around wait 1 s, set
    # the error word and return, and so do the others
    case, fields = W.couette(8, 64)
    ref = T.Lattice(case, fields)
    ref.step(20)
    f_ref, h_ref = ref.populations()
    ref.close()

    lat = T.Lattice(case, fields)
    assert "tclbm_resident" in lat.describe()
    T.tclbm_test_skip_row(lat.handle, 12)
    lat.step(20)
    with pytest.raises(T.TclbmError) as err:
        lat.diagnostics()
    assert err.value.status == T.ETIMEOUT
    T.tclbm_test_skip_row(lat.handle, -1)
    lat.init_fields(fields)
    lat.step(20)
    f, h = lat.populations()
    lat.close()
    assert np.array_equal(f, f_ref) and np.array_equal(h, h_ref)


def test_allocator_returning_null_gives_enomem(T):
    case, _ = W.random_periodic(64, 32, seed=1)
    params = T.params_from_case(case)
    alloc = T.ALLOC_FN(lambda nbytes, stream, ctx: None)
    free = T.FREE_FN(lambda ptr, nbytes, stream, ctx: None)
    with pytest.raises(T.TclbmError) as err:
        T.tclbm_create(params, alloc, free, None, None)
    assert err.value.status == T.ENOMEM


def test_non_finite_state_is_reported(T):
    case, fields = W.random_periodic(64, 32, seed=2)
    fields = {k: np.array(v) for k, v in fields.items()}
    fields["rho"][5, 7] = np.nan
    lat = T.Lattice(case, fields)
    lat.step(2)
    with pytest.raises(T.TclbmError) as err:
        lat.diagnostics()
    assert err.value.status == T.ENONFINITE
    lat.close()


@pytest.mark.parametrize("name,make", [
    ("rb_walls", lambda: W.rayleigh_benard(96, 48, Ra=2e4, seed=11)),
    ("periodic", lambda: W.random_periodic(70, 37, seed=12, force="accel")),
    ("x_ends", lambda: W.with_walls(*W.random_periodic(66, 10, seed=13), axis="x", kind="equilibrium")),
])
def test_resume_from_populations_equals_an_uninterrupted_run(T, name, make):
    # checkpoint = the populations read out; resume = a new handle set from them
    case, fields = make()
    whole = T.Lattice(case, fields)
    whole.step(40)
    f_ref, h_ref = whole.populations()
    whole.close()
    first = T.Lattice(case, fields)
    first.step(17)
    f, h = first.populations()
    first.close()
    second = T.Lattice(case)
    second.set_populations(f, h)
    second.step(23)
    f2, h2 = second.populations()
    second.close()
    assert np.array_equal(f2, f_ref) and np.array_equal(h2, h_ref)


@pytest.mark.parametrize("name,nx,ny,storage", [("chained_sr", 1536, 768, "fp16"), ("tiles", 300, 250, "fp32")])
def test_steps_before_a_failed_launch_count(T, name, nx, ny, storage):
    # the sixth launch of a call fails: five steps are taken and counted, and the lattice goes on
    # from there (with its draws) as one that never saw a failure
    case, fields = W.rayleigh_benard(nx, ny, seed=31, storage=storage)
    case = dict(case, rounding="stochastic" if storage != "fp32" else "nearest")
    lat = T.Lattice(case, fields)
    T.tclbm_test_fail_launch(5)
    with pytest.raises(T.TclbmError) as err:
        lat.step(12)
    T.tclbm_test_fail_launch(-1)
    assert err.value.status == T.ECUDA and lat.steps_done == 5
    lat.step(7)
    got = lat.populations()
    lat.close()
    lat = T.Lattice(case, fields)
    for _ in range(12):
        lat.step(1)
    exp = lat.populations()
    lat.close()
    assert np.array_equal(got[0], exp[0]) and np.array_equal(got[1], exp[1])


def test_batch_steps_before_a_failed_launch_count(T):
    # two kernel groups: the sixth launch is the second group's third step, so the first group
    # has taken three steps, the second and the batch two, and the batch goes on from there
    cases = [W.rayleigh_benard(96, 40, seed=32), W.taylor_green(64, F0=1e-6, nu=0.02)]
    lats = [T.Lattice(c, f) for c, f in cases]
    batch = T.Batch(lats)
    T.tclbm_test_fail_launch(5)
    with pytest.raises(T.TclbmError) as err:
        batch.step(9)
    T.tclbm_test_fail_launch(-1)
    assert err.value.status == T.ECUDA
    assert batch.steps_done == 2 and [lat.steps_done for lat in lats] == [3, 2]
    batch.step(3)
    batch.step(130)
    assert batch.steps_done == 135 and [lat.steps_done for lat in lats] == [136, 135]
    got = [lat.populations() for lat in lats]
    batch.close()
    for (c, f), lat, (gf, gh), n in zip(cases, lats, got, (136, 135)):
        lat.close()
        ref = T.Lattice(c, f)
        ref.set_kernel(1)
        ref.step(n)
        ef, eh = ref.populations()
        ref.close()
        assert np.array_equal(gf, ef) and (gh is None or np.array_equal(gh, eh))
