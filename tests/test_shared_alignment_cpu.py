"""Shared arrays of scalars that the kernels access 8 or 16 bytes at a time
declare that alignment: without it the compiler may place them behind any
other variable, and the wide accesses would be misaligned."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), 'paper_2305_02752_gb300', 'csrc')
DECL = re.compile(r'__shared__\s+(?P<align>__align__\((?P<n>\d+)\)\s+)?(?:unsigned\s+)?(?P<type>[\w:<>]+)\s+(?P<vars>[^;(]*);')
WIDE = {'int2': 8, 'float2': 8, 'int4': 16, 'float4': 16, 'uint4': 16, 'double2': 16}
SCALAR = {'char', 'short', 'int', 'unsigned', 'long', 'float', 'double', 'R', 'T'}


def _kernels(text):
    """The text between one __global__ and the next."""
    parts = text.split('__global__')
    return parts[1:]


def _narrow(text):
    """(array, bytes of an access, declared alignment) of every shared array of
    scalars that is accessed more widely than it is aligned."""
    bad = []
    for body in _kernels(text):
        for d in DECL.finditer(body):
            if d['type'] not in SCALAR:
                continue
            align = int(d['n'] or 0)
            for name in re.findall(r'(\w+)\s*\[', d['vars']):
                sizes = [WIDE[w] for w in re.findall(r'reinterpret_cast<(?:const )?(\w+) \*>\(&?%s\b' % name, body) if w in WIDE]
                sizes += [16 for _ in re.findall(r'(?:load|store)_quad\(%s\b' % name, body)]
                if sizes and max(sizes) > align:
                    bad.append((name, max(sizes), align))
    return bad


def test_finds_a_narrow_array():
    src = '__global__ void k() { __shared__ float s[8]; __shared__ __align__(16) int t[4];\n' \
          ' reinterpret_cast<const float4 *>(s)[0]; store_quad(t, 0, 4, true, q); }'
    assert _narrow(src) == [('s', 16, 0)]


@pytest.mark.parametrize('source', sorted(f for f in os.listdir(CSRC) if f.endswith('.cu')))
def test_wide_shared_arrays_are_aligned(source):
    with open(os.path.join(CSRC, source)) as f:
        assert _narrow(f.read()) == []
