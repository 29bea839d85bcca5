"""The hash that keys bench.py's profiled counters covers every header the kernel
sources include: a change of any of them makes the counters count as outdated."""
import importlib.util
import os
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture()
def bench(tmp_path):
    spec = importlib.util.spec_from_file_location("bench_sources_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    copy = tmp_path / "csrc"
    shutil.copytree(os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"), copy)
    mod.CSRC = str(copy)
    return mod


@pytest.mark.parametrize("sources,headers", [
    (("mixed.cu",), ("dp_internal.cuh", "atom_cta.cuh", "conv.cuh", "tc.cuh")),
    (("embed_x.cu",), ("dp_internal.cuh", "oz.cuh", "tc.cuh")),
    (("embed_cheb.cu", "fit_oz.cu"), ("dp_internal.cuh", "cheb.cuh", "cheb_domain.h", "atom_cta.cuh", "oz.cuh", "tc.cuh")),
])
def test_hash_covers_the_headers(bench, sources, headers):
    before = bench.source_sha(*sources)
    assert bench.source_sha(*sources) == before
    for name in sources + headers:
        path = os.path.join(bench.CSRC, name)
        with open(path) as f:
            text = f.read()
        with open(path, "w") as f:
            f.write(text + "// changed\n")
        assert bench.source_sha(*sources) != before, name
        with open(path, "w") as f:
            f.write(text)
    assert bench.source_sha(*sources) == before
