"""The autotuner against the library it tunes (CPU only): its spaces hold the library's defaults, which are timed first,
and a cached setting counts only for the kernel sources it was tuned on."""
import os
import re
from types import SimpleNamespace

import pytest

from paper_2206_10885_gb300 import autotune as A


def constants():
    with open(os.path.join(A.CSRC, "kns_api.cu")) as f:
        return {k: int(v) for k, v in re.findall(r"constexpr int (k\w+) = (\d+);", f.read())}


@pytest.mark.parametrize("width", [32, 64])
@pytest.mark.parametrize("precision", [0, 1])
def test_the_default_is_in_the_space_and_comes_first(precision, width):
    k, wide = constants(), width == 64
    want = ({"tail_rays": k["kRenderBf16TailRaysWide" if wide else "kRenderBf16TailRays"],
             "bf16_inner_steps": k["kRenderBf16InnerSteps" if wide else "kRenderBf16InnerStepsNarrow"],
             "bf16_min_active": k["kRenderBf16MinActive"]} if precision == 1 else
            {"block_tiles": k["kRenderBlockTiles"], "inner_steps": k["kRenderBlockInnerSteps"],
             "min_active": k["kRenderBlockMinActive"], "static_tiles": k["kRenderStaticTiles"],
             "blocks_per_sm": k["kRenderBlocksPerSM"],
             "tail_rays": k["kRenderBf16TailRays" if wide else "kRenderTailRays"]})
    space = A.space_for(precision)
    assert A.default_setting(precision, width) == want
    assert all(v in space[name] for name, v in want.items())
    cands = A.ordered_candidates(space, precision, width)
    assert cands[0] == want and len(cands) == len(list(A.candidates(space)))


def test_a_space_without_the_default_is_kept_as_given():
    space = {"tail_rays": (-1, 7)}
    assert A.ordered_candidates(space, 0, 32) == list(A.candidates(space))


def test_a_changed_kernel_source_changes_the_cache_key(tmp_path, monkeypatch):
    grid = SimpleNamespace(desc=SimpleNamespace(N=16, sdf_width=32, sdf_hidden=3, pe_pos_L=4, occ_res=128))
    monkeypatch.setattr(A, "CSRC", str(tmp_path))
    source = tmp_path / "kernel.cu"
    keys = []
    for text in ("a", "b", "a"):
        source.write_text(text)
        keys.append(A._key(grid, 1, 64, 64, 128, 0, "GPU"))
    assert keys[0] == keys[2] != keys[1]
