"""Which form of a kernel runs, on both sides of every line between two forms: the tests that compare the
forms with one another (test_gpu_batch_rows, test_gpu_persist_rows, test_gpu_deep_columns) would pass
without comparing anything if both sides ran the same one."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T
from test_gpu_batch_rows import CASES
from test_gpu_deep_columns import _system
from test_gpu_persist_rows import SYSTEMS, _star

pytestmark = pytest.mark.gpu


def _ring(n):
    """n masses on a circle, each joined to the next two."""
    a = np.arange(n) * 2 * np.pi / n
    pos = np.stack([np.cos(a), np.sin(a), np.full(n, 0.5)], 1) * n / 60
    ends = np.array([(i, (i + d) % n) for i in range(n) for d in (1, 2)], np.uint32)
    s = len(ends)
    e = ends.astype(np.int64)
    return inputs.System(pos=pos, vel=np.zeros((n, 3)), mass=np.full(n, 0.1), fixed=np.zeros(n, np.uint8), ends=ends,
                         k=np.full(s, 10.0), rest=np.linalg.norm(pos[e[:, 1]] - pos[e[:, 0]], axis=1),
                         damping=np.full(s, 1.0), dt=1e-4, ground=True, act_amp=np.full(s, 0.1),
                         act_phase=np.linspace(0, 6, s), act_freq=2.0)


@pytest.mark.parametrize("act", [True, False], ids=["actuated", "plain"])
@pytest.mark.parametrize("name", list(CASES))
def test_batches_of_short_rows_start_in_the_row_form(name, act):
    with T.Batch(CASES[name](act)) as b:
        most = 384 if act else 512
        assert b.groups() and all(g["form"] == T.FORM_ROWS and g["launch_threads"] <= most for g in b.groups())
        for g in range(len(b.groups())):
            b.configure(g, 512, 1)
        assert all(g["form"] == T.FORM_PLAIN and g["launch_threads"] == 512 for g in b.groups())


def test_a_system_with_a_longer_row_takes_the_looped_form_beside_the_others():
    with T.Batch([_star(26, 7), _star(27, 8), _ring(300)]) as b:
        form = [b.groups()[b.group_of(r)]["form"] for r in range(3)]
    assert form == [T.FORM_ROWS, T.FORM_PLAIN, T.FORM_ROWS]


def test_the_autotuner_reports_the_form_it_keeps():
    with T.Batch(CASES["clusters_2_3_4"](True)) as b:
        b.autotune(20)
        for g in b.groups():
            assert g["launch_threads"] <= 384 if g["form"] == T.FORM_ROWS else g["launch_threads"] == g["threads"]


@pytest.mark.parametrize("sy,act,per_spring,form", [
    (lambda: SYSTEMS["row_26"](), False, False, T.FORM_ROWS), (lambda: SYSTEMS["row_28"](), False, False, T.FORM_PLAIN),
    (lambda: _star(27, 9), False, False, T.FORM_PLAIN), (lambda: SYSTEMS["cube"](), False, False, T.FORM_ROWS),
    (lambda: SYSTEMS["cube"](), False, True, T.FORM_PLAIN),
    # with the sinusoid from 256 masses on; masses a CTA of at most eight: 384 with actuation, 512 without
    (lambda: _ring(255), True, False, T.FORM_PLAIN), (lambda: _ring(256), True, False, T.FORM_ROWS),
    (lambda: _ring(255), False, False, T.FORM_ROWS),
    (lambda: _ring(384), True, False, T.FORM_ROWS), (lambda: _ring(385), True, False, T.FORM_ROWS),
    (lambda: _ring(3072), True, False, T.FORM_ROWS), (lambda: _ring(3073), True, False, T.FORM_PLAIN),
    (lambda: _ring(512), False, False, T.FORM_ROWS), (lambda: _ring(4096), False, False, T.FORM_ROWS),
    (lambda: _ring(4097), False, False, T.FORM_PLAIN)],
    ids=["row_26", "row_28", "row_27", "cube", "per_spring", "255", "256", "255_plain", "384", "385", "3072", "3073", "512", "4096", "4097"])
def test_persistent_form(sy, act, per_spring, form):
    sy = sy()
    if not act:
        sy.act_amp = None
    if per_spring:
        sy.damping = np.linspace(0.5, 1.5, sy.n_springs)
    with T.Sim(sy, exec_mode=T.EXEC_PERSISTENT) as sim:
        assert sim.exec_mode == T.EXEC_PERSISTENT and sim.step_form == form
        sim.step(3)
        x, _, _ = sim.snapshot()
    assert np.isfinite(x).all()


def test_small_bodies_with_the_worm_take_rows():
    sy = _ring(100)
    amp, sy.act_amp = sy.act_amp, None
    with T.Sim(sy, exec_mode=T.EXEC_PERSISTENT) as sim, T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=1) as ref:
        for s in (sim, ref):
            T.titan_set_worm_actuation(s.handle, np.arange(sy.n_springs), amp, np.linspace(0.0, 0.9, sy.n_springs), 20.0, 0.01)
            s.step(9)
        assert sim.step_form == T.FORM_ROWS
        for s in (sim, ref):                          # and give them up for the sinusoid
            T.titan_set_actuation(s.handle, np.arange(sy.n_springs), amp, np.linspace(0, 6, sy.n_springs), 2.0)
            s.step(9)
        x, y = sim.snapshot(), ref.snapshot()
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])


def test_actuation_set_later_changes_the_form_with_the_entries():
    sy = _ring(3100)                                  # 388 masses a CTA of eight
    amp, phase, sy.act_amp = sy.act_amp, sy.act_phase, None
    with T.Sim(sy, exec_mode=T.EXEC_PERSISTENT) as sim, T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=1) as ref:
        assert (sim.step_form, ref.step_form) == (T.FORM_ROWS, T.FORM_PLAIN)
        for s in (sim, ref):
            s.step(5)
            T.titan_set_actuation(s.handle, np.arange(sy.n_springs), amp, phase, 2.0)
            s.step(9)
        assert sim.exec_mode == T.EXEC_PERSISTENT and sim.step_form == T.FORM_PLAIN
        x, y = sim.snapshot(), ref.snapshot()
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])


@pytest.mark.parametrize("shape,form", [((8 * 76, 8, 16), T.FORM_DEEP), ((8 * 61, 8, 20), T.FORM_PLAIN),
                                         (304 * 256, T.FORM_DEEP), (304 * 256 + 1, T.FORM_PLAIN), (777, T.FORM_DEEP)],
                         ids=str)
def test_step_form(shape, form):
    torch = pytest.importorskip("torch")
    assert torch.cuda.get_device_properties(0).multi_processor_count == 152      # 304 CTAs are two an SM
    sy = _system(shape, True, True, False)
    for variant in (4, 6) if isinstance(shape, tuple) else (4,):
        with T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=variant) as sim:
            assert (sim.csr_kernel, sim.step_form) == (variant, form)
    with T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=1) as sim:
        assert sim.step_form == T.FORM_PLAIN


@pytest.mark.parametrize("n", [100, 600])
def test_actuation_set_again_and_again(n):
    """Every value set is stepped with, also where the plan of the launch stays as it is."""
    sy = _ring(n)
    sy.act_amp = None
    ids, rng = np.arange(sy.n_springs), np.random.default_rng(n)
    with T.Sim(sy, exec_mode=T.EXEC_PERSISTENT) as sim, T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=1) as ref:
        for k in range(6):
            amp, phase = rng.uniform(0, 0.2, sy.n_springs), rng.uniform(0, 6, sy.n_springs)
            for s in (sim, ref):
                if k in (2, 3):
                    T.titan_set_worm_actuation(s.handle, ids, amp, phase / 7, 20.0, 0.01)
                else:
                    T.titan_set_actuation(s.handle, ids, amp, phase, 2.0 + k)
                if k == 4:
                    T.titan_set_spring_params(s.handle, ids[:3], damping=np.array([0.5, 0.7, 1.3]))
                s.step(7)
            x, y = sim.snapshot(), ref.snapshot()
            assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1]), k
        assert sim.exec_mode == T.EXEC_PERSISTENT and sim.step_form == T.FORM_PLAIN        # per-spring damping now
