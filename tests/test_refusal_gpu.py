"""A refused resident handle of many subgames: the message counts the handle's chunks (it is
built before the handle is released), and the autotuner goes on to the layouts that apply."""
import pytest

from paper_2605_19928_gb300 import capi, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()
    capi.use_torch_allocator()


def test_refused_batch_names_its_chunks():
    specs = synth.batch_rivers(256, n_hands=48)
    with pytest.raises(capi.CfrError, match=r"\(512 chunks") as e:  # 48 hands: two chunks of 32
        capi.cfr_batch_create(specs, capi.make_opts("dcfr", schedule="resident"))
    assert e.value.code == capi.CFR_EINVAL
    best, ms = capi.cfr_autotune(specs, capi.make_opts("dcfr", precision="single"), iters=2)
    assert best.schedule != capi.CFR_SCHEDULE_RESIDENT and ms > 0
