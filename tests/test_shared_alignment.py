"""Static shared-memory arrays that a kernel reads or writes through a wider type are declared with that type's alignment
(the language gives an array the alignment of its elements and no more).  Read off the sources; no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_10183_b200", "csrc")
BYTES = {"uint8_t": 1, "uint16_t": 2, "__half": 2, "__half2": 4, "float": 4, "int": 4, "uint32_t": 4, "uint64_t": 8, "float2": 8, "uint2": 8,
         "float4": 16, "uint4": 16}


def _functions(text):
    """The pieces of a file from one function with static shared arrays to the next."""
    starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
    return [text[a:b] for a, b in zip(starts, starts[1:])]


def test_wide_accesses_to_static_shared_arrays_are_aligned():
    seen, wrong = 0, []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        for body in _functions(open(os.path.join(CSRC, name)).read()):
            for m in re.finditer(r"(?<!extern )__shared__ (?:__align__\((\d+)\) )?(\w+) (\w+)\[", body):
                have = max(int(m.group(1) or 0), BYTES.get(m.group(2), 8))
                for wide in re.findall(r"reinterpret_cast<(?:const )?(\w+)\*>\(&?%s\b" % m.group(3), body):
                    seen += 1
                    if BYTES[wide] > have:
                        wrong.append(f"{name}: {m.group(3)} is {have}-byte aligned and accessed as {wide}")
    assert seen >= 3  # (the scan finds what it is meant for)
    assert not wrong, "\n".join(sorted(set(wrong)))
