"""The one-kernel decode form's histogram bins (csrc/decode_coop.cuh: key_bin): ordered like the values, no wider than a
quarter of an octave at any magnitude in use, and narrow where thresholds lie."""
import os
import re
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09323_b200", "csrc")


def _keys(g):
    """gate_key of finite values (moc_common.cuh)."""
    b = (np.asarray(g, np.float32) + np.float32(0)).view(np.uint32)
    return np.where(b >> 31 != 0, ~b, b | np.uint32(1 << 31))


def _values(keys):
    with np.errstate(invalid="ignore"):
        g = np.where(keys >> 31 != 0, keys & np.uint32(0x7fffffff), ~keys).view(np.float32)
    return np.where(np.isfinite(g), g, np.float32(0))


def test_bins(tmp_path):
    text = open(os.path.join(CSRC, "decode_coop.cuh")).read()
    code = re.search(r"constexpr int kBins.*?static_assert.*?\n", text, re.S).group(0).replace("__host__ __device__", "")
    source, program = tmp_path / "bins.cpp", tmp_path / "bins"
    source.write_text("#include <cstdint>\n#include <cstdio>\n" + code + "int main() { uint32_t k; std::printf(\"%d\\n\", kBins); "
                      "while (std::fread(&k, 4, 1, stdin) == 1) std::printf(\"%u\\n\", key_bin(k)); }")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", str(source), "-o", str(program)], check=True)
    rng = np.random.default_rng(2)
    steps = np.arange(2048, dtype=np.uint64) << 21   # the key steps of a quarter of an octave: first, second, last key of each
    edges = np.concatenate([steps, steps + 1, steps + (1 << 21) - 1]).astype(np.uint32)
    normal = {std: _keys(rng.standard_normal(11008) * std + mean) for std, mean in
              ((1.28, 0.0), (0.4, 0.0), (0.013, 0.0), (1e-6, 0.0), (1e4, 0.0), (1.0, -1.5))}
    keys = np.sort(np.concatenate([edges, rng.integers(0, 2 ** 32, 40000, dtype=np.uint32), *normal.values()]))
    out = subprocess.run([str(program)], input=keys.tobytes(), check=True, capture_output=True).stdout.split()
    bins = np.array(out[1:], np.int64)
    assert bins.min() >= 0 and bins.max() < int(out[0])
    assert (np.diff(bins) >= 0).all()
    of = dict(zip(keys.tolist(), bins.tolist()))
    g = np.abs(_values(keys))
    in_use = (g >= 2.0 ** -24) & (g < 2.0 ** 14)
    steps = (np.diff(keys >> 21) > 0) & in_use[1:] & in_use[:-1]
    assert steps.sum() > 300 and (np.diff(bins)[steps] > 0).all()   # two quarters of an octave do not share a bin
    for std, k in normal.items():
        k = np.sort(k)[::-1]
        for kept in (688, 1376, 2752):
            shared = sum(of[v] == of[k[kept - 1]] for v in k.tolist())
            assert shared <= (40 if 0.1 < std < 2 and k[kept - 1] >= 1 << 31 else 1000), (std, kept, shared)
