"""A committed traffic figure names every source file that its kernels are compiled from, and drops out
when any of them changes."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2501_07047_gb300", "csrc")


def bench():
    spec = importlib.util.spec_from_file_location("hefx_bench_profiles", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("kernel,sources", [("ntt_cc", ["ntt_cc_impl.cuh"]),
                                            ("ntt_cc_2p", ["ntt_cc_2p.cuh", "ntt_cc_impl.cuh"])])
def test_any_source_of_the_kernels_counts(kernel, sources, tmp_path):
    b = bench()
    figures = [b.profile_traffic(kernel, w) for w in ("fwd", "inv")]
    assert None not in figures
    (tmp_path / "profiles").mkdir()
    (tmp_path / "paper_2501_07047_gb300" / "csrc").mkdir(parents=True)
    name = os.path.join("profiles", kernel + "_traffic.txt")
    (tmp_path / name).write_text(open(os.path.join(ROOT, name)).read())
    copies = [tmp_path / "paper_2501_07047_gb300" / "csrc" / s for s in sources]
    for c in copies:
        c.write_bytes(open(os.path.join(CSRC, c.name), "rb").read())
    b.ROOT = str(tmp_path)
    assert [b.profile_traffic(kernel, w) for w in ("fwd", "inv")] == figures
    for c in copies:
        kept = c.read_bytes()
        c.write_bytes(kept + b"// changed\n")
        assert b.profile_traffic(kernel, "fwd") is None, c.name
        c.write_bytes(kept)
