"""What the device code's types refuse, by the CUDA compiler's front end (no GPU)."""
import os
import subprocess

import pytest

from paper_1511_02166_gb300 import build


def front_end(tmp_path, source):
    """The compiler's messages for a translation unit that includes the solver."""
    src = tmp_path / "probe.cu"
    src.write_text('#include "%s"\nnamespace panel {\n%s\n}\n'
                   % (os.path.join(build.CSRC, "k_solve_mixed.cu"), source))
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", os.path.join(build.ROOT, "include"), "-c", str(src), "-o",
                        str(tmp_path / "probe.o")], capture_output=True, text=True)
    return r.returncode, r.stdout + r.stderr


@pytest.mark.parametrize("rhs,res", [("ClusterRhs", "float"), ("IrRhs", "float"),
                                     ("SmemRhs", "double")])
def test_row_sums_refuse_a_temporary_right_hand_side(tmp_path, rhs, res):
    """RowSums keeps a reference to its right-hand side until finish(): one built from a
    temporary reads a dead object.  Both assertions below have to fail to hold: the
    compiler stops at them, before any code generation."""
    rc, out = front_end(tmp_path, """
    using Sums = RowSums<ResAcc, {rhs}, {res}>;
    static_assert(std::is_constructible<Sums, {rhs}, {res}*, int, int, int>::value, "refuses rvalue");
    static_assert(std::is_constructible<Sums, const {rhs}, {res}*, int, int, int>::value,
                  "refuses const rvalue");
    static_assert(!std::is_constructible<Sums, const {rhs}&, {res}*, int, int, int>::value,
                  "takes lvalue");
    """.format(rhs=rhs, res=res))
    assert rc != 0
    for what in ("refuses rvalue", "refuses const rvalue", "takes lvalue"):
        assert 'failed with "%s"' % what in out, out
    assert "3 errors detected" in out, out
