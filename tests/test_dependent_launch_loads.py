"""Kernels are resident before the kernels whose words they read have finished, so
those words are not read through the non-coherent path: in the device sources it is
used for the twiddle tables alone.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_04510_gb300", "csrc")


def code():
    """{file: source without comments}"""
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*")):
        if path.endswith((".cu", ".cuh", ".h")):
            out[os.path.basename(path)] = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    return out


def test_non_coherent_loads_are_for_static_tables():
    src = code()
    nc = {f: re.findall(r"ld\.global\.nc|__ldg\s*\(|\bldu\.", s) for f, s in src.items()}
    assert {f for f, m in nc.items() if m} == {"he_internal.h"} and len(nc["he_internal.h"]) == 1
    body = src["he_internal.h"].split("ulonglong2 ld2_static(", 1)[1].split("\n}", 1)[0]
    assert "ld.global.nc" in body
    users = {f: re.findall(r"ld2_static\(([^;]*);", s) for f, s in src.items() if f != "he_internal.h"}
    assert {f for f, m in users.items() if m} == {"ntt.cu"} and len(users["ntt.cu"]) == 1
    # the one caller, ld_tw, is given entries of a twiddle table
    tw = re.findall(r"(?<!ulonglong2 )\bld_tw\(([^;]*);", src["ntt.cu"])
    assert tw and all(a.startswith("tw_entry<") for a in tw)
