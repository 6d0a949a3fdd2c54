"""The tuner times schedules on operands laid out as the calls lay theirs out:
one function gives both the row stride, and it is the one whose rows a call's
workspace holds."""
import os

import pytest

nt = pytest.importorskip("paper_2307_16080_gb300.nk_tune")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_16080_gb300", "csrc")


@pytest.mark.parametrize("name,calls", [("tune.cu", "const int64_t ld = tc_operand_ld(kind, K);"),
                                        ("nk_api.cu", "P.ldk = tc_operand_ld(kind, P.K);")])
def test_one_row_stride(name, calls):
    assert calls in open(os.path.join(CSRC, name)).read()


@pytest.mark.parametrize("prec,esz,parts", [("bf16", 2, 1), ("fp8", 1, 1), ("bf16x3", 2, 2)])
@pytest.mark.parametrize("K", [1, 100, 255, 256, 257, 1001])
def test_workspace_holds_rows_of_that_stride(prec, esz, parts, K):
    ld = -(-K // 16) * 16 if K < 256 else -(-K // (128 // esz)) * (128 // esz)
    rows = 4096   # both operands, in every part
    one, two = (nt.nk_workspace_size(nt.matmul_problem(M, 2048, K, prec), (128, 128, 128 // esz, 1, 3, 1))
                for M in (2048, 2048 + rows))
    assert two - one == rows * ld * esz * parts
