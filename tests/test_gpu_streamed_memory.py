"""What an out-of-core render allocates for its chunks is given back (needs a GB300)."""
import numpy as np
import pytest
import torch

from paper_1606_04427_gb300 import build, render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("vector", [False, True])
def test_streamed_render_frees_every_chunk(vector):
    ps = synth.two_species_set(30000, 12000, 6, grid=64).with_brightness([0.05, 0.3])
    if vector:  # a chunk then holds an emission per particle as well
        ps.rgb = np.random.default_rng(2).uniform(0.1, 1.0, (42000, 3)).astype(np.float32)
        ps.col_vector = np.array([0, 1], np.int32)
    base = render.torch_allocator()
    held = {}

    def alloc(n, stream):
        p = base._alloc_py(n, stream)
        held[p] = n
        return p

    def free(p, stream):
        del held[p]
        base._free_py(p, stream)

    render.render_streamed(ps, synth.front_camera(160, 120), 10000, allocator=render.CallbackAllocator(alloc, free))
    torch.cuda.synchronize()
    assert held == {}
