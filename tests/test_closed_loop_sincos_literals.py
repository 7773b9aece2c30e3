"""The closed loop's copy of the sine and cosine coefficients (csrc/closed_loop.cu)
is the one derived by sincos_coeffs.py, highest degree first: sin a = a + a z P(z),
cos a = 1 + z (-1/2 + z Q(z)), z = a^2."""
import os
import re

import pytest

pytest.importorskip("mpmath")

from paper_1507_04769_gb300 import sincos_coeffs as sc  # noqa: E402

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1507_04769_gb300", "csrc", "closed_loop.cu")


def _table(name):
    text = open(SRC).read()
    body = text[text.index(f"double {name}[7] = {{"):]
    body = body[body.index("{") + 1:body.index("}")]
    return [float.fromhex(v) if "0x" in v else float(v) for v in re.split(r",\s*", body.strip())]


def test_literals_are_the_derived_coefficients():
    P, Q, _, _ = sc.coefficients()
    assert _table("kClSin") == [0.0] + list(P[::-1])
    assert _table("kClCos") == list(Q[::-1]) + [-0.5]
