"""The passes' other forms compile without register spills too, at the registers that their blocks per SM
leave (ptxas resource usage; no GPU needed)."""
from concurrent.futures import ThreadPoolExecutor

import pytest

from test_build_resources import _nvcc, _resources

# part of the mangled name -> (source, registers per thread that the launch bound leaves)
FORMS = {
    "8k_updateILi0ELb1E": ("gi_cache.cu", 40),  # GI_MERGE_WARP
    "13k_update_listILi0ELb0E": ("gi_cache.cu", 40),
    "13k_update_listILi0ELb1E": ("gi_cache.cu", 40),
    "16k_update_batchedILi0E": ("gi_cache.cu", 40),
    "15k_resolve_denseE": ("gi_cache.cu", 64),
    "8k_filterE": ("gi_probes.cu", 64),
    "9k_projectE": ("gi_probes.cu", 128),
    "11k_reprojectE": ("gi_probes.cu", 64),
    "8k_gatherE": ("gi_probes.cu", 64),
    "17k_gather_temporalE": ("gi_probes.cu", 64),
    "21k_interpolate_batchedE": ("gi_probes.cu", 48),
    "k_nrc_encodeILi0E": ("gi_nrc.cu", 40),
    "k_nrc_encodeILi1E": ("gi_nrc.cu", 40),
    "k_nrc_encode_queriesE": ("gi_nrc.cu", 48),
    "k_nrc_selectE": ("gi_nrc.cu", 40),
    "k_nrc_inferE": ("gi_nrc.cu", 128),
    "k_nrc_adamILi64E": ("gi_nrc.cu", 64),
    "k_nrc_adamILi256E": ("gi_nrc.cu", 64),
}


def test_other_forms_do_not_spill(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    sources = sorted({src for src, _ in FORMS.values()})
    with ThreadPoolExecutor(len(sources)) as ex:
        found = dict(zip(sources, ex.map(lambda s: _resources(nvcc, s, str(tmp_path)), sources)))
    for key, (src, most) in FORMS.items():
        names = [n for n in found[src] if key in n]
        assert names, f"{key} not compiled from {src}"
        for n in names:
            assert found[src][n]["spill"] == 0, f"{n} spills {found[src][n]['spill']} bytes"
            assert found[src][n]["regs"] <= most, f"{n} uses {found[src][n]['regs']} registers"
