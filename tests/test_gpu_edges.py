"""Inputs at the edges of what the entry points take, and calls whose speed or
memory need rests on a rule: each was wrong, refused or slow once.  Results are
whole numbers and are compared with the oracle for equality."""
import numpy as np
import pytest

from gpu_helpers import gpu_select
from helpers import layer_z, make_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_1810_11966_gb300 as jp
    jp.load(build_if_missing=True)
    return jp


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("up,down", [(2**31 - 1, -2), (2**31 - 2, -3), (2**30, -2**30 - 1)])
def test_offsets_whose_differences_wrap(lib, oracle_mod, mode, up, down):
    # decreasing offsets whose 32-bit differences are all positive: refused
    # wherever they lie (PAPER mode reads the last station only), in both forms
    ev = [[(0.1 * z, 0.2 * z, z)] * 2 for z in layer_z(2)]
    good = make_batch([ev] * 3, 2)
    assert np.all(np.diff(np.array([0, up, down, 6], np.int32)) > 0)
    for at in (1, 4, 7, 10):
        off = good["offsets"].copy()
        off[at], off[at + 1] = up, down
        b = dict(good, offsets=off)
        assert oracle_mod.run(oracle_mod.params(2, mode, t_xz=0.25), b)["status"] != 0
        ctx = lib.Context(lib.params(2, mode, t_xz=0.25))
        for form in ("plain", "batched"):
            assert gpu_select(ctx, b, form=form, triplets=False)["status"] == lib.JPSI_EINVAL, (at, form)
        ctx.close()
