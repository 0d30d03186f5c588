"""A tune cache written when other kernels stood behind the choices is not used: its lines have no kernel generation in
their keys (or another one), so the layers are timed again and the file gets lines of this generation."""
import re

import pytest

from workloads import workload
from oracle import problem as oprob
from tests.gpu_helpers import engine_args_from_oracle

pytestmark = pytest.mark.gpu


def test_choices_of_replaced_kernels_are_timed_again(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    w = workload("xyz3_onebath", K=4)
    chains, mpos = engine_args_from_oracle(oprob.build_inputs(w))

    def routes(path):
        eng = capi.Engine(chains, mpos, chi_max=w.chi_max, eps=w.eps, max_steps=w.K, autotune=True, tune_cache=str(path))
        r = eng.routes()
        eng.destroy()
        return r

    new, old = tmp_path / "new.tsv", tmp_path / "old.tsv"
    assert not any(r[3] for r in routes(new).values())
    keys = [ln.split("\t")[0] for ln in open(new)]
    with open(old, "w") as f:
        for key in keys:
            f.write(re.sub(r"\|g\d+$", "", key) + "\t2\t1\n")
            f.write(re.sub(r"\|g\d+$", "|g1", key) + "\t2\t1\n")
    assert not any(r[3] for r in routes(old).values())
    assert all(r[3] for r in routes(old).values())            # the second time from this generation's lines
