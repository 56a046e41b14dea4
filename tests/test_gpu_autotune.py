"""The autotuner's cache: one entry per kind of batch, and a choice of an older build's movers is
not taken over without a measurement."""
import json

import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def tune(ion_nstep=1):
    phys = W.bounded_small(ncells=128, ppc=50, seed=15, ion_nstep=ion_nstep)
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=-1, block=0)
    sim.load_all(W.initial_load(phys, seed=15))
    sim.step(400)
    sim.sync()
    sim.close()


@pytest.fixture
def cache(tmp_path, monkeypatch):
    ensure_built()
    path = tmp_path / "tune.json"
    monkeypatch.setenv("BITPIC_TUNE_CACHE", str(path))
    return path


def test_subcycled_batches_have_their_own_entry(cache):
    tune()
    tune(ion_nstep=4)
    assert len(json.loads(cache.read_text())) == 2


def test_an_older_builds_choice_is_measured_anew(cache):
    tune()
    (key, choice), = json.loads(cache.read_text()).items()
    # the key as builds wrote it before it named the movers and the subcycling
    gpu, *rest = key.split("|")
    old = "|".join([gpu] + [r for r in rest if r in ("fp32", "fp64", "mag", "nomag") or r[0] in "pc"])
    assert old != key
    cache.write_text(json.dumps({old: [512, 80]}))
    tune()
    entries = json.loads(cache.read_text())
    assert entries.pop(old) == [512, 80]
    (block, sort), = entries.values()
    assert block in (128, 256, 512) and sort in (10, 20, 40, 80)
