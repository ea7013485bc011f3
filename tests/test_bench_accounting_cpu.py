"""The byte accounting of bench.py: in every launch form each band's coefficients belong to one kernel per direction, and
counters captured from other kernels are not printed as those of the present ones."""
import json
import os

import pytest

import bench
import workloads as wl
from helpers import library_plan

FROM = "bands_from_spectrum/"


@pytest.mark.parametrize("name, forms", [
    ("config2", ["class0", "class1", "class2", "class3", "class4"]),
    ("config1", ["chirp", "merged", "class0"]),
    ("config2", ["split", "merged", "class0"]),
    ("table1", ["pow2", "class0"]),
    ("config4", ["class0", "class1", "class2", "class3", "class4"]),
    ("config2", ["class0/smooth", "class1/smooth", "class2/smooth", "class3", "class4/smooth"]),
    ("table1", ["pow2", "class0/smooth"]),
])
def test_every_band_belongs_to_one_kernel(name, forms):
    w = wl.CONFIGS[name]
    plan = library_plan(w, device=-1)
    names = [FROM + f for f in forms] + ["bands_to_spectrum/" + f for f in forms]
    names += ["band2p_cols/analysis/large", "band2p_rows/analysis/large", "band2p_cols/synthesis/large", "band2p_rows/synthesis/large"]
    owned = bench.kernel_algorithmic_bytes(plan, w, 3, names)
    assert set(n for n in owned if "bands_" in n) <= set(names)
    assert all(owned.get(n, 0) > 0 for n in names if "bands_" in n)
    assert sum(owned.values()) == bench.path_algorithmic_bytes(plan, w, 3)
    plan.close()


def test_directions_may_differ_in_the_kernel_of_a_class():
    w = wl.CONFIGS["config2"]
    plan = library_plan(w, device=-1)
    names = [FROM + f"class{c}/smooth" for c in (0, 1, 2, 4)] + [FROM + "class3"] + [f"bands_to_spectrum/class{c}" for c in range(4)] + ["bands_to_spectrum/class4/smooth"]
    owned = bench.kernel_algorithmic_bytes(plan, w, 3, names)
    assert {n for n in owned if "bands_" in n} == set(names)
    assert sum(owned.values()) == bench.path_algorithmic_bytes(plan, w, 3)
    plan.close()


def test_captured_counters_name_the_sources_they_belong_to():
    captured = json.load(open(os.path.join(bench.ROOT, "profiles", "dram_traffic_workload2.txt")))
    assert len(captured["kernel_sources"]) == len(bench.kernel_source_digest()) == 16
    assert set(captured["config2"]) == {"rfft_cols_fwd", "rfft_rows_fwd", "irfft_rows", "irfft_cols"} | {
        f"bands_{d}_spectrum/class{c}" for d in ("from", "to") for c in range(5)}
