"""The forms of the slab phases, run on the host.

transform_forms.cu compiles the phases' own source for the host without
contraction and compares, bit for bit, the compiled-in plans with the run-time
ones and rows shared by a block with rows of a warp, for every two-radix plan.  It
also holds the FP64 slab plans of every pair of padded lengths to the share of
lanes that their z transforms keep busy."""
import os
import subprocess

from paper_2208_01348_gb300 import build as b


def test_forms_of_the_transform_phases_agree(tmp_path):
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path / "transform_forms")
    cmd = [b._nvcc()] + b.GENCODE + ["-O0", "-Xcompiler", "-ffp-contract=off", "-std=c++17",
                                     "--expt-relaxed-constexpr", "-diag-suppress", "20208", "-I" + b.SRC,
                                     "-I" + os.path.join(b.ROOT, "include"), os.path.join(here, "transform_forms.cu"),
                                     os.path.join(b.SRC, "slab_plan.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
