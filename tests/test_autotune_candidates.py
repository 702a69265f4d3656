"""The autotuner times each choice of kernels once: no two candidates differ only in a value
that selects nothing (the FP64 panel width outside the DFMA form, the assembly chunk of
uniform meshes), and choices cached when the values selected something else are not used."""
import pytest


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("order", [0, 1, 2, 3, 4])
def test_candidates_select_different_kernels(precision, order):
    from paper_1605_01020_gb300 import autotune
    cands = autotune.candidates(precision, order)
    kernels = [(c["lu_persistent"], c["lu_tensor"], c["lu_panel"] if precision == 0 and c["lu_tensor"] == 0 else None,
                c["asm_chunk"] if order == 0 else None) for c in cands]
    assert len(set(kernels)) == len(kernels)
    forms = {0: {0, 1}, 1: {0, 1, 2}, 2: {1}, 3: {1}}[precision]
    assert {c["lu_tensor"] for c in cands} == forms
    assert all(c["asm_chunk"] in ((8, 16, 32) if order == 0 else (0,)) for c in cands)


def test_earlier_cache_entries_are_not_used():
    from paper_1605_01020_gb300 import autotune

    class Mesh:
        d, order, Np = 3, 3, 64
    assert autotune.mesh_key(Mesh, 0, "gpu") != "gpu|d3|p3|Np64|prec0"
