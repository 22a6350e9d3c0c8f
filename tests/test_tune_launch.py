"""The launch tuners on a stand-in batch whose step time is a table by option:
they end no slower than the library's own choice, set no solve blocks before
their turn (the automatic choice cannot be asked for again), and spend no steps
on options that have no effect."""
import pytest

from paper_2503_05046_gb300 import native, tune

AUTO = 8  # blocks per scene that the library takes by itself here


class FakeBatch:
    def __init__(self):
        self.options, self.seen = {}, []

    def set_option(self, option, value):
        self.options[option] = value

    def synchronize(self, stats=True):
        pass

    def seconds(self):
        self.seen.append(dict(self.options))
        blocks = self.options.get(native.BATCH_OPT_SOLVE_BLOCKS, AUTO)
        g2p = self.options.get(native.BATCH_OPT_G2P_THREADS, 256)
        return {1: 4.27, 2: 2.65, 4: 1.99, 8: 1.71}[blocks] + {128: 0.0, 256: 0.1, 512: 0.2}[g2p]


@pytest.fixture
def batch(monkeypatch):
    b = FakeBatch()
    monkeypatch.setattr(tune, "_time_batch", lambda batch, h, n, solver, steps: batch.seconds())
    return b


def test_tuned_batch_is_no_slower_than_untouched(batch):
    untouched = batch.seconds()
    best, table = tune.tune_batch_launch(batch, 1e-4, 4, None)
    assert batch.seconds() <= untouched
    assert best[native.BATCH_OPT_SOLVE_BLOCKS] == 8 and best[native.BATCH_OPT_G2P_THREADS] == 128
    assert min(t for _, t in table) == pytest.approx(1.71)


def test_solve_blocks_stay_the_librarys_until_their_turn(batch):
    tune.tune_batch_launch(batch, 1e-4, 4, None)
    first = next(i for i, o in enumerate(batch.seen) if native.BATCH_OPT_SOLVE_BLOCKS in o)
    others = [o for o in batch.seen if native.BATCH_OPT_SOLVE_BLOCKS not in o]
    assert first == len(others)
    for knob, values in ((native.BATCH_OPT_G2P_THREADS, {128, 256, 512}),
                         (native.BATCH_OPT_GRID_PARTICLES, {512, 2048, 8192})):
        assert {o.get(knob) for o in others} >= values


def test_no_steps_for_options_without_effect(batch, monkeypatch):
    best, table = tune.tune_batch_launch(batch, 1e-4, 4, None)
    assert len({o.get(native.BATCH_OPT_P2G_CHUNK) for o in batch.seen}) == 1
    assert len(table) == 3 + 3 + 4  # G2P threads, grid particles, solve blocks
    assert best[native.BATCH_OPT_P2G_CHUNK] == 256  # (named all the same, as ever)
    assert tune.tune_batch.__defaults__[1] == (256,)

    class Sim:
        ctx, scene = None, {"h": 1e-4, "substeps": 10}

    def no_step(*a, **k):
        raise AssertionError("a step for nothing")
    options = []
    monkeypatch.setattr(native, "mpm_step", no_step)
    monkeypatch.setattr(native, "mpm_set_option", lambda ctx, o, v: options.append((o, v)))
    (form, chunk), table = tune.tune_p2g_form(Sim(), None)
    assert (form, chunk) == (0, 256) and table == []
    assert options == [(native.OPT_P2G_FORM, 0), (native.OPT_P2G_CHUNK, 256)]
