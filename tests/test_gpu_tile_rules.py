"""Parity at the edges of the kernel-selection rules: tile widths, remainders and splits that only some shapes reach."""
import numpy as np
import pytest

from paper_2108_13342_b200 import binding as B
from paper_2108_13342_b200 import workloads as W
from util import RTOL_BF16, RTOL_F32, check, close, graph, rnd, run_both

pytestmark = pytest.mark.gpu
FUSED = B.PLAN_FUSED


def _bf(x):
    return W.round_to_bf16(x)


def gemm(m, n, k, epi, kmajor_b=False, seed=900):
    g = graph()
    g.ext("A", (m, k), "bf16")
    ins = {"A": _bf(rnd((m, k), seed, -1, 1))}
    if kmajor_b:
        g.ext("Bt", (n, k), "bf16"); ins["Bt"] = _bf(rnd((n, k), seed + 1, -0.1, 0.1))
        b = g.add("Transpose", ["Bt"], perm=(1, 0))
    else:
        g.ext("Bm", (k, n), "bf16"); ins["Bm"] = _bf(rnd((k, n), seed + 1, -0.1, 0.1)); b = "Bm"
    t = g.add("MatMul", ["A", b])
    if epi != "none":
        g.ext("bias", (n,), "f32"); ins["bias"] = rnd((n,), seed + 2, -0.5, 0.5)
        t = g.add("Add", [t, "bias"])
    if epi == "bias_gelu":
        t = g.add("Gelu", [t], approx="tanh")
    if epi == "bias_residual":
        g.ext("R", (m, n), "bf16"); ins["R"] = _bf(rnd((m, n), seed + 3, -1, 1))
        t = g.add("Add", [t, "R"])
    g.mark_output(t)
    return W.Workload(g, ins)


@pytest.mark.parametrize("mnk", [(4000, 760, 200), (4096, 768, 72), (4096, 584, 1032)])
@pytest.mark.parametrize("kmajor_b", [False, True])
@pytest.mark.parametrize("epi", ["none", "bias_gelu", "bias_residual"])
def test_pair_gemm_192_columns(mnk, kmajor_b, epi):
    """CTA-pair kernel with 192-column tiles: each CTA's half of B is one and a half 64-column boxes, each epilogue warp's
    part three 32-column chunks; ragged last tile in both directions."""
    m, n, k = mnk
    s = check(gemm(m, n, k, epi, kmajor_b), RTOL_BF16, FUSED | B.PLAN_NO_TILE_GEMM, expect_blocks=1)
    b = s.g.blocks()[0]
    assert b["variant"] == 3 and b["grid"] == 2 * ((m + 255) // 256) * ((n + 191) // 192), b
