"""Kernels' function attributes are set for the device of every handle, not once per process: they belong
to a device's context, and a handle on a second device would otherwise fail at its first launch.  (Checked
in the sources: the tests run on one device.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_11169_gb300", "csrc")


def source(name):
    return open(os.path.join(CSRC, name)).read()


def test_no_attribute_behind_a_process_wide_flag():
    for name in sorted(os.listdir(CSRC)):
        s = source(name)
        if "cudaFuncSetAttribute" in s:
            assert not re.search(r"once_flag|call_once|static bool", s), name


def test_creation_sets_them_all():
    create = source("api.cpp").split("icwf_status icwf_create(")[1].split("\nicwf_status ")[0]
    declared = set(re.findall(r"cudaError_t (\w+_attributes)\(\);", source("icwf_internal.h")))
    assert declared and all(f + "()" in create for f in declared)
    # what the kernel files of a handle define is declared there
    defined = set()
    for name in os.listdir(CSRC):
        if name.endswith(".cu") and name != "exact2d.cu":
            defined |= set(re.findall(r"^cudaError_t (\w+_attributes)\(\) \{", source(name), re.M))
    assert {d for d in defined if d != "propagate_attributes"} == declared
