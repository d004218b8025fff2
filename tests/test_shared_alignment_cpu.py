"""A shared-memory array that is read or written by vectors has to be declared with
their alignment: the compiler places an array of 4-byte words on any multiple of 4,
and a 16-byte access off a multiple of 16 is a fault. Checked on the sources."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_02346_gb300", "csrc")
VECTOR = r"(?:u?int2|u?int4|float2|float4|ulonglong2|double2)"
DECL = re.compile(r"__shared__\s+(?!__align__|alignas)(?:const\s+)?(float|uint32_t|int|unsigned|uint16_t|__nv_bfloat16|uint8_t)"
                  r"\s+(\w+)\s*\[")


def misdeclared(text):
    """Names of shared arrays of scalars, declared without an alignment, that the
    same kernel reads through a pointer to vectors."""
    bad = []
    for body in re.split(r"(?=__global__)", text):
        for _, name in DECL.findall(body):
            if re.search(rf"reinterpret_cast<\s*(?:const\s+)?{VECTOR}\s*\*\s*>\(\s*&?{name}\b", body):
                bad.append(name)
    return bad


def test_the_check_itself():
    use = "{ auto q = reinterpret_cast<const float4*>(sw)[1]; }"
    assert misdeclared("__global__ void k() { __shared__ float sw[256]; " + use) == ["sw"]
    assert not misdeclared("__global__ void k() { __shared__ __align__(16) float sw[256]; " + use)
    assert not misdeclared("__global__ void k() { __shared__ float4 sw[64]; " + use)


def test_sources():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    assert {f: b for f in files for b in [misdeclared(open(f).read())] if b} == {}
