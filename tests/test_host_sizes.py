"""Host-side sizes of device workspaces, from the headers that the kernels'
launchers use (a small program compiled with nvcc and run on the host: no GPU).
"""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_05125_gb300 import build as B


def run_host(tmp_path, source, data=""):
    """compile `source` against the package's headers; its output as words"""
    try:
        nvcc = B._nvcc()
        subprocess.run([nvcc, "--version"], check=True, capture_output=True)
    except (OSError, RuntimeError, subprocess.CalledProcessError):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "host.cu", tmp_path / "host"
    src.write_text(source)
    inc = os.path.join(os.path.dirname(B.HERE), "include")
    subprocess.run([nvcc, *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", inc, str(src), "-o",
                    str(exe)], check=True)
    return subprocess.run([str(exe)], input=data, check=True, capture_output=True, text=True).stdout.split()


def test_sort_counters_fit_every_smaller_count(tmp_path):
    # a volume's build scratch is cut once, for the most triangles seen, and
    # any smaller count is sorted in it: the counters that a sort of m keys
    # lays out (two counts per tile and digit, then a total per digit) have to
    # lie inside those of every n >= m
    n = np.unique(np.concatenate([[1, 2, 1023, 1024, 1025, 2047, 2048, 2049, 4097], np.arange(480_000, 1_100_000, 509),
                                  (1 << 19) + np.arange(-2050, 2051, 41), (1 << 20) + np.arange(-2, 3), [3_250_000, 1 << 24]]))
    out = run_host(tmp_path, """
        #include <cstdio>
        #include "bvh.cuh"
        int main()
        {
            unsigned long long n;
            while (std::scanf("%llu", &n) == 1) {
                const size_t used = 512 * adgi::radix_tiles(n) + 256;
                std::printf("%zu %zu %zu\\n", used, adgi::radix_hist_entries(n), adgi::bvh_scratch_layout_bytes(n));
            }
        }""", "\n".join(map(str, n)))
    used, held, layout = np.array(out, np.int64).reshape(-1, 3).T
    assert len(used) == len(n)
    assert (np.maximum.accumulate(used) <= held).all()
    assert (np.diff(held) >= 0).all() and (np.diff(layout) >= 0).all()


def test_stand_in_stays_inside_the_samples(tmp_path):
    # a Metropolis sample takes the hit and record of the sample whose ray
    # equals its own; a word that names none of the n samples (an old sort key
    # left where inconsistent offsets made the kernel drop a range) is not an
    # index, and the sample keeps its own
    out = run_host(tmp_path, """
        #include <cstdio>
        #include "kernels.cuh"
        int main()
        {
            const unsigned n = 1000u, words[] = {0u, 1u, 998u, 999u, 1000u, 1001u, 0x7FFFFFFFu, 0x80000000u, 0xFFFFFFFFu};
            for (unsigned q : {0u, 17u, 999u})
                for (unsigned w : words) std::printf("%u %u %u\\n", q, w, adgi::stand_in(w, q, n));
        }""")
    q, word, got = np.array(out, np.int64).reshape(-1, 3).T
    np.testing.assert_array_equal(got, np.where(word < 1000, word, q))
