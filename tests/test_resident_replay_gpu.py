"""Iterations of the resident schedule captured into a user's graph and replayed."""
import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, synth
from test_gpu_parity import _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["pairs", "single"])
@pytest.mark.parametrize("alternating", [True, False])
def test_replayed_launches_continue_the_solve(alternating, precision):
    import torch
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.use_torch_allocator()
    spec = synth.river_subgame(n_hands=203, seed=3, range_seed=4)
    opts = capi.make_opts("dcfr", precision=precision, alternating=alternating, schedule="resident")
    stream = torch.cuda.Stream()
    states = []
    for replayed in (False, True):
        tree = capi.cfr_batch_create([spec], opts, stream=stream.cuda_stream)
        try:
            capi.cfr_iterate(tree, 2)
            if replayed:
                capi.cfr_sync(tree)
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    capi.cfr_iterate(tree, 3)
                with torch.cuda.stream(stream):
                    for _ in range(4):
                        graph.replay()
            else:
                capi.cfr_iterate(tree, 12)
            capi.cfr_sync(tree)
            states.append(_state(tree, 1))
        finally:
            capi.cfr_tree_destroy(tree)
    def same(a, b):
        if isinstance(a, dict):
            assert a.keys() == b.keys()
            for k in a:
                same(a[k], b[k])
        elif isinstance(a, (list, tuple)):
            assert len(a) == len(b)
            for x, y in zip(a, b):
                same(x, y)
        else:
            assert np.array_equal(np.asarray(a), np.asarray(b))
    same(states[0], states[1])
