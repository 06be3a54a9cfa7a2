"""Batch.launches_per_step against the launches a batch queues."""
import pytest

from paper_2101_07163_gb300 import lbmice
from tests.captured import launched

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,shapes,one,two", [
    ("f32", [0] * 3, 1, 1),                  # march members, in pairs
    ("f32", [0, 0, 1], 2, 3),                # a tile shape takes two launches for two steps
    ("f32", [0] * 65 + [1, 2], 4, 6),        # 64 + 1 march members in two launches
    ("bf16", [0, 0, 1], 2, 4),
])
def test_launches_of_one_step_and_of_two(storage, shapes, one, two):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = lbmice.Batch([dict(nx=40, ny=36, storage=storage)] * len(shapes), stream=st)
        for i, (m, s) in enumerate(zip(b.members, shapes)):
            m.init_seed(20, 18, 6.0, 0.3)
            b.set_shape(i, s)
        b.sync()
    assert b.launches_per_step == one
    assert len(launched(st, lambda: b.step(1))) == one
    assert len(launched(st, lambda: b.step(2))) == two
    b.close()
