"""That the cases of the kernel comparisons do take the path they are about:
the divided pass is one launch more than the undivided one that kernel timing
takes, and the kernel on bulk-copied tiles is the one whose waits the test hook
makes run out."""
import pytest

import test_split_gpu
import test_tma_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("name", sorted(test_split_gpu.CASES))
def test_divided_pass_runs(name, prec):
    from paper_1407_4524_gb300 import lbm
    dom = lbm.Domain(dict(test_split_gpu.CASES[name], lattice="D3Q19", precision=prec), device=0)
    dom.step(1)
    divided = dom.launches_per_step()
    dom.set_kernel_timing(True)
    assert divided == dom.launches_per_step() + 1
    dom.close()


@pytest.mark.parametrize("name", sorted(test_tma_gpu.CASES))
def test_kernel_on_bulk_copied_tiles_runs(name, monkeypatch):
    from paper_1407_4524_gb300 import lbm
    monkeypatch.setenv("LBM_STAGED_TEST_EXPIRE", "1")
    dom = lbm.Domain(dict(test_tma_gpu.CASES[name], precision="fp16"), device=0)
    dom.step(1)
    assert dom.stats()["timeouts"] != 0
    dom.close()
