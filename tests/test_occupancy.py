"""Registers and shared memory of kernels that lost CTAs per SM to code of other forms, as the
compiler reports them."""
import os
import re
import subprocess

import pytest

from paper_1303_0008_gb300 import build as B

LINEAR, SQRT, CONJ, GENW = range(4)


@pytest.fixture(scope="module")
def ctas(tmp_path_factory):
    """ctas(file, kernel): the CTAs of 256 threads that an SM holds, by its 65536 registers and
    227 KB of shared memory."""
    d = tmp_path_factory.mktemp("ptxas")
    known = {}

    def load(name):
        try:
            nvcc = B.nvcc()
        except RuntimeError:  # pragma: no cover
            pytest.skip("needs nvcc")
        r = subprocess.run([nvcc, *B.ARCH, *B.FLAGS, "-Xptxas", "-v", "-c",
                            os.path.join(B.CSRC, name), "-o", str(d / "out.o")],
                           capture_output=True, text=True, check=True)
        out, entry = {}, None
        for line in r.stderr.splitlines():
            m = re.search(r"Compiling entry function '(\S+)'", line)
            if m:
                entry = m.group(1)
            m = re.search(r"Used (\d+) registers", line)
            if m and entry:
                shared = re.search(r"(\d+) bytes smem", line)
                regs = 256 * 8 * -(-int(m.group(1)) // 8)
                smem = 1024 + (int(shared.group(1)) if shared else 0)
                out[entry] = min(65536 // regs, 227 * 1024 // smem, 8)
        return out

    def of(name, kernel, mode=None):
        if name not in known:
            known[name] = load(name)
        tag = f"{len(kernel)}{kernel}" + (f"ILi{mode}EE" if mode is not None else "E")
        found = [v for k, v in known[name].items() if tag in k]
        assert len(found) == 1, (kernel, mode)
        return found[0]

    return of


@pytest.mark.parametrize("kernel,mode,least", [
    ("k_smooth_colour64", GENW, 8), ("k_residual64", GENW, 6), ("k_residual_restrict64", GENW, 4),
    ("k_defect64", GENW, 6), ("k_fas_rhs64", GENW, 8), ("k_smooth_colour64", LINEAR, 5),
    ("k_residual64", LINEAR, 5), ("k_residual_restrict64", LINEAR, 4),
    ("k_smooth_colour64", SQRT, 3), ("k_residual_restrict64", SQRT, 2)])
def test_one_form_does_not_carry_the_others(ctas, kernel, mode, least):
    assert ctas("mg_fp64.cu", kernel, mode) >= least


@pytest.mark.parametrize("kernel,least", [
    ("kb_smooth64", 3), ("kb_smooth_tile64", 4), ("kb_residual_restrict64", 2),
    ("kb_residual_restrict_tile64", 2), ("kb_fas_rhs64", 3), ("kb_fas_rhs_tile64", 4),
    ("kb_handoff64", 2), ("kb_handoff_tile64", 4), ("kb_prolong64", 6), ("kb_prolong_column64", 3),
    ("kb_prolong32", 8), ("kb_prolong_column32", 5), ("kb_residual_restrict32", 3),
    ("kb_smooth32", 5)])
def test_batch_stages_in_tiles_and_cell_by_cell(ctas, kernel, least):
    assert ctas("mg_batch.cu", kernel) >= least
