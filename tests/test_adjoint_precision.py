"""The adjoint of the outlet row divides by the density with a rounded
quotient, as the forward step does (an approximate one differs by less than
any gradient test could see, so the source is read for it)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05158_gb300", "csrc")


def test_the_outlet_row_takes_a_rounded_quotient():
    src = open(os.path.join(CSRC, "lbm_channel.cu")).read()
    body = re.search(r"void fold_outlet\((.*?)\n}\n", src, re.S).group(1)
    assert "const float ir = __fdiv_rn(1.f, rho);" in body and "__fdividef" not in body
    assert not re.search(r"\bir\b", body.split(") {")[0])  # nor is a quotient handed in
