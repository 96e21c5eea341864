"""Reciprocals and square roots of the device code are CUDA's own functions
(correctly rounded over the whole range, subnormals and infinities too), not
sequences of approximate instructions. Read from the sources."""
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_01975_gb300", "csrc")


def test_no_approximate_instructions():
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        for word in ("rcp.approx", "rsqrt.approx", "sqrt.approx", "div.approx", "div.full", "ex2.approx", "lg2.approx"):
            assert word not in text, (name, word)
