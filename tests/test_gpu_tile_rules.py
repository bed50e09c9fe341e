"""Parity at the edges of the kernel-selection rules: tile widths, remainders and splits that only some shapes reach."""
import numpy as np
import pytest

from paper_2108_13342_b200 import binding as B
from paper_2108_13342_b200 import workloads as W
from util import RTOL_BF16, RTOL_BF16_ROUNDING, RTOL_F32, check, close, graph, rnd, run_both

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


@pytest.mark.parametrize("rows,cols", [(1, 33), (5000, 7), (3, 129), (40000, 31), (1200, 128), (1184, 197), (1183, 257), (9, 538), (2368, 511),
                                       (700, 1025), (64, 2047), (30, 4095), (5, 5001)])
@pytest.mark.parametrize("kind", ["softmax", "layernorm", "interpreted"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_rows_that_fit_no_vector(rows, cols, kind, dtype):
    """Row blocks whose length is no multiple of four: every lane count and warp split of the element-wise form, with a
    compile-time chain and an interpreted one."""
    g = graph()
    g.ext("X", (rows, cols), dtype)
    x = rnd((rows, cols), 910, -2, 2)
    ins = {"X": _bf(x) if dtype == "bf16" else x}
    if kind == "layernorm":
        g.ext("ga", (cols,)); g.ext("be", (cols,))
        ins.update(ga=rnd((cols,), 911, 0.5, 1.5), be=rnd((cols,), 912, -0.5, 0.5))
        y = g.add("LayerNorm", ["X", "ga", "be"], axis=-1, eps=1e-5)
    else:
        y = g.add("Softmax", [g.add("MulC", ["X"], c=0.5) if kind == "softmax" else g.add("Sigmoid", ["X"])], axis=-1)
    g.mark_output(y)
    check(W.Workload(g, ins), RTOL_F32 if dtype == "f32" else RTOL_BF16_ROUNDING, expect_blocks=1)
