"""Device memory of a default FP64 hierarchy: five vectors per level (a third more for the
coarser ones), the Krylov basis and a few work vectors; not the patch corrections (51
numbers per vertex, 5.7 vectors), which only the split and the per-patch sweeps use."""
import pytest

pytestmark = pytest.mark.gpu


def test_patch_corrections_are_allocated_where_they_are_used():
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    n = 512
    vec = 8 * stokes.vec_len(n)
    stokes.stokes_test_set_alloc_limit(int(14.5 * vec))
    try:
        pkg.Hierarchy(n, restart=1).close()
        for kw in ({"tile": 4}, {"tile": 5}):
            with pytest.raises(stokes.StokesError) as err:
                pkg.Hierarchy(n, restart=1, **kw)
            assert err.value.status == stokes.STOKES_ERR_OOM
    finally:
        stokes.stokes_test_set_alloc_limit(0)
    pkg.Hierarchy(n, restart=1, tile=4).close()
