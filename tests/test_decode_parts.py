"""The one-kernel decode form's parts of the narrow bins (csrc/decode_coop.cuh): the part that a key is counted in is one of its own bin's, in
the order of the values, and the limit that a settled part gives is the least key of that part."""
import os
import re
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09323_b200", "csrc")
FROM, TO = 0xbd000000, 0xc1800000   # keys of 2^-5 and 2^4


def test_parts_belong_to_their_bin(tmp_path):
    text = open(os.path.join(CSRC, "decode_coop.cuh")).read()
    code = re.search(r"constexpr int kBins.*?static_assert\(narrow_bins_follow.*?\n", text, re.S).group(0).replace("__host__ __device__", "")
    source, program = tmp_path / "parts.cpp", tmp_path / "parts"
    source.write_text("#include <cstdint>\n#include <cstddef>\n#include <cstdio>\n" + code + "int main() { std::printf(\"%u %u %d\\n\", kFineFrom, kFineTo, "
                      "kNarrowBins); uint32_t k; while (std::fread(&k, 4, 1, stdin) == 1) std::printf(\"%u\\n\", narrow_bin(key_bin(k))); }")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", str(source), "-o", str(program)], check=True)
    rng = np.random.default_rng(3)
    starts = np.arange(FROM, TO, 1 << 16, dtype=np.uint64)
    keys = np.sort(np.concatenate([starts, starts + 0xffff, rng.integers(FROM, TO, 20000, dtype=np.uint64)])).astype(np.uint32)
    first, *bins = subprocess.run([str(program)], input=keys.tobytes(), check=True, capture_output=True, text=False).stdout.decode().splitlines()
    assert first.split() == [str(FROM), str(TO), str((TO - FROM) >> 16)]
    bins = np.array(bins, np.int64)
    for parts in (8, 16, 32, 64, 128, 256):
        shift = 16 - int(np.log2(parts))
        counter = (keys.astype(np.int64) - FROM) >> shift           # as the kernel counts
        least = FROM + (counter << shift)                           # as it gives the limit
        assert (counter // parts == bins).all()                     # a bin's counters are its own
        assert (np.diff(counter) >= 0).all()
        assert (least <= keys).all() and (keys < least + (1 << shift)).all()
