"""The phases of the matvec and D-hat transforms, run on the host.

transform_phases.cu compiles the phases' own source for the host and compares
every two-radix plan (all padded lengths up to 256, forward and inverse, FP32
and FP64, full, ragged and one-cell lines) with sums of roots of unity, the
x pass with its symmetric product, the D-hat build's even and odd lines, and
the slab plans of every pair of padded lengths with the limits of a block.
The bounds, 4 eps per radix-2 level of each transform in the relative 2-norm,
follow from the number of roundings per element."""
import os
import subprocess

from paper_2208_01348_gb300 import build as b


def test_transform_phases_match_sums_of_roots_of_unity(tmp_path):
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path / "transform_phases")
    cmd = [b._nvcc()] + b.GENCODE + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-diag-suppress", "20208",
                                     "-I" + b.SRC, "-I" + os.path.join(b.ROOT, "include"),
                                     os.path.join(here, "transform_phases.cu"), os.path.join(b.SRC, "slab_plan.cu"),
                                     "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
