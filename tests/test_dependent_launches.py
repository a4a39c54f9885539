"""Loads of kernels that start before the kernel ahead of them has ended
(launch_next in csrc/internal.h).  A non-coherent load (__ldg) needs data that
nothing writes while its kernel is resident: in these kernels only what is laid
down when a handle is created, never a table of powers."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1201_0499_gb300", "csrc")


def source(name):
    return open(os.path.join(CSRC, name)).read()


def test_values_kernel_reads_only_lists_and_coefficients_non_coherently():
    text = source("kernels_sum.cu")
    fixed = {"co", "sp.fac", "sp.poly_ptr", "sp.act_bits", "sp.act", "hq", "sp.hits"}
    assert re.search(r"\*co = reinterpret_cast<const int4 \*>\(sp\.coef ", text)
    assert re.search(r"\*hq = sp\.hit_ptr ", text)
    bases = {m.strip() for m in re.findall(r"__ldg\(([\w.]+)", text)}
    assert bases and bases <= fixed, bases - fixed


def test_flagged_point_kernels_read_the_table_coherently():
    for name, read_only in (("kernels.cu", "A::load_full"), ("kernels_wide.cu", "wide::load_wf"),
                            ("kernels_qd.cu", "qd::load_wf")):
        uses = [line for line in source(name).splitlines() if re.search(re.escape(read_only) + r"\(", line)]
        uses = [u for u in uses if "pp.points" not in u and "coef" not in u]  # inputs and coefficients
        assert uses and all("kSome ?" in u for u in uses), (name, uses)
