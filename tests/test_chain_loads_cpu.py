"""Band kernels that run as members of a chain read what earlier kernels wrote without a wait of their own, so those loads
have to be the ones that the L1 does not serve (band_common.cuh).  Checked on the source: a kernel that can be in a chain
uses no other load for the spectrum or the coefficients, and one that waits for itself keeps the ordinary ones."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_29119_b200", "csrc")


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", ["band_analysis.cu", "band_synthesis.cu", "band_pow2.cu", "band_chirp.cu", "band_split.cu", "band_smooth.cuh"])
def test_chained_kernels_load_past_the_l1(name):
    s = code(name)
    assert not re.search(r"\bld_data\s*\(|__ldc[sgav]\s*\(|__ldlu\s*\(", s)
    # __ldg and plain subscripts are for plan tables and shared memory: never on the spectrum, the coefficients or the planes
    assert not re.search(r"__ldg\s*\(\s*(Xs?|c|in|Ys?|out)\b", s)
    assert not re.search(r"=\s*\*?\b(Xs?|c|in|Ys)\s*\[", s)
    assert re.search(r"\bld_chained\s*\(|\bld_spectrum<CHAINED>|\bld_coefficient<CHAINED>", s)


def test_the_load_itself_is_strong_at_device_scope():
    body = re.search(r"float2 ld_chained\(.*?\n}", code("engine.cuh"), re.S).group(0)
    assert "asm volatile" in body and "ld.relaxed.gpu.global" in body
    common = code("band_common.cuh")
    assert re.search(r"ld_spectrum\([^)]*\)\s*{\s*return CHAINED \? ld_chained\(p\)", common)
    assert re.search(r"ld_coefficient\([^)]*\)\s*{\s*return CHAINED \? ld_chained\(p\)", common)
    assert "ld_spectrum<CHAINED>(X" in common and "ld_data(X" not in common     # slot_value
    for name in ("band_pow2.cu", "band_chirp.cu", "band_split.cu"):   # always members or heads
        assert "slot_value<true>(" in code(name) and "slot_value<false>(" not in code(name)
    # whole-CTA class kernels and the two-pass kernels are in no chain
    for name in ("band_analysis.cu", "band_synthesis.cu"):
        assert re.search(r"if constexpr \(W == 0\) return generic \|\| chained \? nullptr", code(name))


def test_only_members_of_a_chain_load_past_the_l1():
    """The kernels of 5-smooth lengths exist in both forms for class 0, which alone is ever in a chain; what a launch gets follows
    from its place in the chain.  (Loads past the L1 in every class cost 1 - 2 % of the large calls, see band_common.cuh.)"""
    from paper_2609_29119_b200 import build
    smooth = code("band_smooth.cuh")
    assert not re.search(r"\bld_chained\s*\(", smooth)
    assert len(re.findall(r"\b(?:ld_spectrum|ld_coefficient|slot_value)<CHAINED>\s*\(", smooth)) == 3
    built = [tuple(int(f[-1]) for f in flags) for _, _, flags in build.VARIANTS]
    assert all(h == 0 for c, _, h in built if c > 0)
    assert all((0, a, h) in built for a in (0, 1) for h in (0, 1))
    listed = re.search(r"#define CQT_SMOOTH_KERNELS\(X\)((?:.*\\\n)*.*)", smooth).group(1)
    as_int = {"false": 0, "true": 1}
    assert sorted(built) == sorted((int(c), as_int[a], as_int[h]) for c, a, h in re.findall(r"X\((\d), (\w+), (\w+)\)", listed))
    assert re.search(r"kernel_of\(analysis, cls, b\.chain == kChainMember\)", code("band_smooth.cu"))
