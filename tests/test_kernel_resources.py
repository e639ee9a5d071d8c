"""What the compiler gives kernels whose speed hangs on it: registers per thread, from the compiler's own report."""
import os
import re
import subprocess

import pytest

from paper_2304_14698_b200 import build


@pytest.fixture(scope="module")
def registers(tmp_path_factory):
    """Registers of a source file's kernels, by their demangled names up to the arguments."""
    done = {}

    def of(source):
        if source not in done:
            out = str(tmp_path_factory.mktemp("ptxas") / "k.o")
            r = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o", out],
                               capture_output=True, text=True)
            assert r.returncode == 0, r.stderr
            found = re.findall(r"Compiling entry function '(\w+)'.*?Used (\d+) registers", r.stderr, re.S)
            names = subprocess.run(["c++filt"], input="\n".join(n for n, _ in found), capture_output=True, text=True).stdout
            done[source] = {n.replace("(anonymous namespace)::", "").split("(")[0].split("::")[-1]: int(v)
                            for n, (_, v) in zip(names.splitlines(), found)}
        return done[source]
    return of


@pytest.mark.parametrize("T,most", [("float", 86), ("__nv_bfloat16", 88)])
@pytest.mark.parametrize("K", [4, 8, 16])
def test_sums_without_stored_rows_carry_nothing_of_the_stores(registers, T, K, most):
    """The last attention layer fused with Eq. 8 (variant 1): a choice made per row took it to 88 and 92 registers and its
    launch over 36 k rows from 14.9 to 16.0 us."""
    assert registers("k_agg_tma.cu")[f"k_aggregate_tma<{T}, {K}, 1, false, false>"] <= most


@pytest.mark.parametrize("kernel,ctas", [("k_embed<__nv_bfloat16, 8, 1>", 3), ("k_embed<__nv_bfloat16, 16, 1>", 3),
                                         ("k_embed<__nv_bfloat16, 32, 1>", 3), ("k_embed<__nv_bfloat16, 32, 2>", 2),
                                         ("k_embed<float, 16, 1>", 2), ("k_embed<float, 32, 1>", 2)])
def test_node_update_of_many_operators_keeps_its_resident_ctas(registers, kernel, ctas):
    """CTAs of 256 threads per SM, whose 65,536 registers are handed out to warps in pieces of 256: the wait for the launch before
    took a third CTA (bf16, hidden 64 and 128, 179 k rows: 59.8 -> 65.9 and 166.5 -> 171.9 us)."""
    per_warp = -(-32 * registers("k_rows.cu")[kernel] // 256) * 256
    assert 65536 // (8 * per_warp) >= ctas
