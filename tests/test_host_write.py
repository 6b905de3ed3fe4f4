"""Whether a kernel may write a caller's host buffer, from what the driver says of its address: the decision by itself."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09800_b200", "csrc")
PAGE = 0x7F0000000000
CASES = [                                                    # type, device's address, range, access, address, bytes -> may write
    ("whole", (1, PAGE, PAGE, 65536, 3, PAGE, 65536), 1),
    ("inside", (1, PAGE + 800, PAGE, 65536, 3, PAGE + 800, 64736), 1),
    ("nothing of it", (1, PAGE, PAGE, 65536, 3, PAGE, 0), 1),
    ("one byte past its end", (1, PAGE, PAGE, 65536, 3, PAGE, 65537), 0),
    ("only its beginning registered", (1, PAGE + 65528, PAGE, 65536, 3, PAGE + 65528, 800), 0),
    ("larger than any range", (1, PAGE + 8, PAGE, 65536, 3, PAGE + 8, 2**64 - 8), 0),
    ("before the range", (1, PAGE - 8, PAGE, 65536, 3, PAGE - 8, 8), 0),
    ("registered for reading", (1, PAGE, PAGE, 65536, 1, PAGE, 64), 0),
    ("no access", (1, PAGE, PAGE, 65536, 0, PAGE, 64), 0),
    ("not aligned", (1, PAGE + 4, PAGE, 65536, 3, PAGE + 4, 64), 0),
    ("another address on the device", (1, PAGE + 4096, PAGE, 65536, 3, PAGE, 64), 0),
    ("not registered", (0, 0, 0, 0, 0, PAGE, 64), 0),
    ("device memory", (2, PAGE, PAGE, 65536, 3, PAGE, 64), 0),
]


@pytest.fixture(scope="module")
def decide(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_write")
    src = d / "decide.cc"
    src.write_text('#include "host_write.h"\n#include <stdlib.h>\n'
                   'int main(int, char **v) { auto u = [&](int k) { return strtoull(v[k], nullptr, 10); };\n'
                   '  hbf::HostMemory m{(uint32_t)u(1), u(2), u(3), (size_t)u(4), u(5)};\n'
                   '  return hbf::device_may_write(m, (const void *)(uintptr_t)u(6), (size_t)u(7)) ? 1 : 0; }\n')
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(d / "decide")])
    return lambda args: subprocess.call([str(d / "decide")] + [str(a) for a in args])


@pytest.mark.parametrize("name, args, expected", CASES, ids=[c[0] for c in CASES])
def test_decision(decide, name, args, expected):
    assert decide(args) == expected
