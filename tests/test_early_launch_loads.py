"""Kernels that are launched before the kernel in front of them has ended
(launch_pdl) read that kernel's results with ordinary loads: the read-only path
(ld.global.nc, __ldg, loads that a const __restrict__ pointer allows to be
moved) is for memory that nothing writes while the kernel runs."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2511_22460_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    src = re.sub(r"//[^\n]*", "", src)
    return re.sub(r"/\*.*?\*/", "", src, flags=re.S)


def test_forward_scan_reads_terms_and_wide_scores_with_ordinary_loads():
    src = _code("ebr_forward.cu")
    assert "ld.global.nc" not in src
    assert not re.search(r"__ldg\(\s*&?a\.(wq|wide_in|route|fx_word|hist|ctrl)\b", src)


def test_early_kernels_take_no_restrict_pointer_to_the_results_before():
    for name, kern, args in (("ebr_fused.cu", "k_pack", ("w", "wmax_bits", "route")),
                             ("ebr_query.cu", "k_final_select", ("keys", "ctrl"))):
        head = re.search(r"\b%s\(([^{;]*?)\)\s*\{" % kern, _code(name)).group(1)
        for a in args:
            assert re.search(r"\*\s*%s\b" % a, head), (kern, a)
            assert not re.search(r"__restrict__\s+%s\b" % a, head), (kern, a)


def test_block_wise_scan_reads_terms_and_wide_scores_with_ordinary_loads():
    src = _code("ebr_fused.cu")
    assert "ld.global.nc" not in src
    assert not re.search(r"__ldg\(\s*&?a\.(wq|wide_in|route|fx_word|hist|ctrl)\b", src)
