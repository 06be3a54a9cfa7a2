"""The form a batched launch takes: by what the launch carries, so that the trials of one size class
alone, single steps and pairs each fill the GPU. The bits of every form are those of single grids
(test_two_step_gpu.py, test_two_step_forms_gpu.py)."""
import pytest

from paper_2101_07163_gb300 import lbmice
from tests.captured import launched

pytestmark = pytest.mark.gpu

MARCH, TILE, TWO_MARCH, TWO_TILE = ("batch_march_kernel", "batch_step_kernelILi32ELi8E",
                                    "batch_two_kernel", "batch_two_tile_kernel")


@pytest.mark.parametrize("sides,flow,storage,one,two", [
    ([64] * 4, False, "f32", [TILE], [TWO_TILE]),
    ([64] * 4, True, "f32", [TILE], [TWO_TILE]),
    ([848], True, "f32", [TILE], [TWO_TILE]),            # 719,104 of 720,896 nodes
    ([850], True, "f32", [MARCH], [TWO_TILE]),
    ([1024], False, "f32", [TILE], [TWO_TILE]),          # 2^20 nodes
    ([1024, 8], False, "f32", [TILE], [TWO_MARCH]),
    ([1024, 1024], False, "f32", [MARCH], [TWO_MARCH]),
    ([1024] + [100] * 63 + [40] * 3, True, "f32", [MARCH, TILE], [TWO_MARCH, TWO_TILE]),
    ([64] * 4, True, "f16", [MARCH], [MARCH, MARCH]),    # 16-bit batches: single steps
], ids=["small", "small_flow", "most_single_tiles_flow", "march_flow", "most_tiles", "two_march",
        "march", "two_launches", "f16"])
def test_form_of_a_launch(sides, flow, storage, one, two):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = lbmice.Batch([dict(nx=n, ny=n, flow=flow, nu=0.05, storage=storage) for n in sides],
                         stream=st)
        for m in b.members:
            m.init_seed(m.nx / 2, m.ny / 2, 5.0, 0.3)
        b.sync()
        for steps, want in ((1, one), (2, two)):
            names = launched(st, lambda: b.step(steps))
            assert len(names) == len(want) and all(w in n for w, n in zip(want, names)), names
        b.close()


def test_a_narrow_member_steps_in_pairs_with_the_others():
    # on its own a grid of 27 columns takes single steps
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = lbmice.Batch([dict(nx=nx, ny=ny, flow=True, nu=0.05) for nx, ny in ((27, 9680), (64, 64))],
                         stream=st)
        for m in b.members:
            m.init_seed(m.nx / 2, m.ny / 2, 5.0, 0.3)
        b.sync()
        names = launched(st, lambda: b.step(2))
        assert len(names) == 1 and TWO_TILE in names[0], names
        b.close()


@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_single_steps_of_a_tuned_batch_do_not_lose_to_a_tile_shape(flow):
    # four grids of 64^2: 4.0 us a step in 32 x 8 tiles (4.9 with flow), 18.8 (21.6) in a march
    import torch

    def batch(shape):
        b = lbmice.Batch([dict(nx=64, ny=64, flow=flow, nu=0.05)] * 4)
        for i, m in enumerate(b.members):
            m.init_seed(32, 32, 8.0, 0.3)
            b.set_shape(i, shape)
        return b

    def us(b):
        best = float("inf")
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(100):
                b.step(1)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]) * 10)
        return best

    march, tile = batch(0), batch(1)
    assert us(march) < 1.5 * us(tile)
    march.close()
    tile.close()
