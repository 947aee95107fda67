"""The persistent kernel's block shape (host side): the library's choice by size, a
caller's shape for every size, and back."""
import pytest

from paper_1502_02908_gb300 import binding as B


@pytest.fixture(autouse=True)
def _auto():
    B.batch_shape_auto()
    yield
    B.batch_shape_auto()


@pytest.mark.parametrize("worth", [0, 1, 303, 304, 305, 40_000])
def test_library_choice_and_callers_shape(worth):
    auto = (256, 1) if worth <= 304 else (256, 2)
    assert B.debug_batch_shape(worth, 152) == auto
    for shape in B.BATCH_SHAPES:
        B.batch_shape(*shape)
        assert B.debug_batch_shape(worth, 152) == shape
    with pytest.raises(B.SimError):
        B.batch_shape(384, 1)
    assert B.debug_batch_shape(worth, 152) == B.BATCH_SHAPES[-1]      # a refused one changes nothing
    B.batch_shape_auto()
    assert B.debug_batch_shape(worth, 152) == auto


def test_tuner_leaves_the_choice_to_the_library_by_default():
    import inspect
    from paper_1502_02908_gb300 import autotune

    class Sim:
        def set_group_threshold(self, x): pass
        def tune(self, x): pass
        def set_launch(self, x): pass

    assert inspect.signature(autotune.autotune).parameters["shapes"].default == (None,)
    best = dict(group_threshold=-1, warp_threshold=-1, launch="persistent", batch_shape=(128, 4))
    autotune.apply(Sim(), best)
    assert B.debug_batch_shape(1, 152) == (128, 4)
    autotune.apply(Sim(), dict(best, batch_shape=None))
    assert B.debug_batch_shape(1, 152) == (256, 1)
