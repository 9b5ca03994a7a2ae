"""Which executor a served request runs on (rcm_serve_policy.hpp), compiled for the host and asked directly:
the decision shows only in a request's latency, never in its result."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_08128_gb300", "csrc")


@pytest.fixture(scope="module")
def cluster(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("policy")
    src = d / "policy.cpp"
    src.write_text('#include "rcm_serve_policy.hpp"\n#include <cstdio>\nint main() { long long n, m; int l, b, x;\n'
                   'while (std::scanf("%lld %d %lld %d %d", &n, &l, &m, &b, &x) == 5)\n'
                   'std::printf("%d\\n", rcm::serve_cluster(n, l, m, b, x)); }\n')
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(d / "policy")], check=True)

    def ask(*rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([str(d / "policy")], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]

    return ask


def test_a_lone_large_request_gets_a_cluster(cluster):
    # vertices, requests in the server, options (least vertices, CTAs), largest cluster of the device
    assert cluster((900_000, 1, 0, 0, 16), (600_000, 1, 0, 0, 16), (524_288, 8, 0, 0, 16), (524_287, 1, 0, 0, 16)) == [8, 8, 8, 0]


def test_under_load_only_the_largest_do(cluster):
    assert cluster((900_000, 9, 0, 0, 16), (1_048_575, 200, 0, 0, 16), (1_048_576, 9, 0, 0, 16), (4_000_000, 64, 0, 0, 16),
                   (4_000_000, 65, 0, 0, 16), (1_048_576, 4000, 0, 0, 16)) == [0, 0, 8, 8, 4, 4]


def test_options_and_devices(cluster):
    assert cluster((300_000, 1, 1 << 18, 0, 16), (300_000, 500, 1 << 18, 0, 16), (300_000, 500, 1 << 18, 6, 16),
                   (900_000, 1, 1 << 20, 6, 16), (4_000_000, 1, -1, 0, 16), (4_000_000, 1, 0, 6, 0)) == [8, 4, 6, 0, 0, 0]
