"""The device code asks for approximate arithmetic by CUDA's own functions and
operators, whose meaning the toolkit states, never by an instruction of its own."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_05047_gb300", "csrc")


def test_no_approximate_instruction_is_spelled_out():
    for path in glob.glob(os.path.join(CSRC, "*")):
        if os.path.isfile(path):
            found = re.findall(r"\b(?:rcp|div|sqrt|rsqrt|ex2|lg2|sin|cos|tanh)\.approx[.\w]*", open(path).read())
            assert not found, (path, found)
