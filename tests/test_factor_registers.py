"""CTAs per SM of the 2D factorisation as the compiler leaves them room: registers of each form of
k_factor_simt times its threads, out of an SM's 65536.  Up to 96 nodes (blocked) and in the column by
column form two CTAs share an SM; wider blocked forms are alone on theirs."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_01467_gb300", "csrc")
# (type, register rows per lane): threads, CTAs per SM
FORMS = {("float2", 2): (256, 2), ("float2", 3): (256, 2), ("float2", 4): (512, 1),
         ("float2", 6): (384, 1), ("float2", 0): (512, 2), ("double2", 0): (512, 2)}


def test_two_ctas_share_an_sm(tmp_path):
    from paper_1909_01467_gb300 import build
    r = subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xptxas", "-v", "-c",
                        os.path.join(CSRC, "factor.cu"), "-o", str(tmp_path / "f.o")], check=True,
                       capture_output=True, text=True)
    found = {}
    for m in re.finditer(r"Compiling entry function '\S*k_factor_simtI\d(\w+?2)Li(\d)E.*?"
                         r"Used (\d+) registers", r.stdout + r.stderr, re.S):
        found[m[1], int(m[2])] = int(m[3])
    assert set(found) == set(FORMS)
    for form, regs in found.items():
        threads, ctas = FORMS[form]
        assert ctas * threads * ((regs + 7) // 8 * 8) <= 65536, (form, regs)
