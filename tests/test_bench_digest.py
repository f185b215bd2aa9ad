"""The digest that guards the bench's measured DRAM traffic covers every file
that launches a kernel inside a product, on CPU: each launcher that device.h
declares after the product's arguments is defined in one of the hashed files."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1412_1756_gb300", "csrc")


def test_digest_covers_every_product_kernel():
    header = open(os.path.join(CSRC, "device.h")).read()
    product = header[header.index("struct ProductArgs"):]
    launchers = set(re.findall(r"\b(launch_\w+)\(", product))
    assert {"launch_core", "launch_near_tile", "launch_receive_tile", "launch_translate_quad"} <= launchers
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            text = open(os.path.join(CSRC, f)).read()
            defined = {n for n in launchers if re.search(r"^cudaError_t " + n + r"\([^;]*\)\s*\{", text, re.M)}
            assert not defined or f in bench.PRODUCT_SOURCES, (f, defined)
            launchers -= defined
    assert not launchers, launchers
