"""The traffic figures that bench.py reports are tied to the sources of the
kernels they were captured on: every file that defines one of those kernels,
or code that it inlines, is in the digest."""
import importlib.util
import pathlib
import re

ROOT = pathlib.Path(__file__).resolve().parents[1]
CSRC = ROOT / "paper_1707_02244_gb300" / "csrc"


def _bench():
    spec = importlib.util.spec_from_file_location("bench_module", ROOT / "bench.py")
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_digest_covers_the_pass_kernels(tmp_path, monkeypatch):
    bench = _bench()
    # where the column and mid pass, their epilogues and their FFT are defined
    defs = (r"col_kernel\(const KParams", r"mid_kernel\(const KParams", r"\bcol_body\(const KParams",
            r"\bmid_body\(const KParams", r"struct EpiAdmm\b", r"void stage_twiddle\(", r"struct KParams \{")
    files = {f.name for f in CSRC.iterdir() if f.is_file() for d in defs if re.search(d, f.read_text())}
    assert {"cs_col.cuh", "cs_mid.cuh", "cs_passes.cuh", "cs_fft.cuh", "cs_internal.h"} <= files
    # a change in any of them changes the digest
    copy = tmp_path / "paper_1707_02244_gb300" / "csrc"
    copy.mkdir(parents=True)
    for f in CSRC.iterdir():
        if f.is_file():
            (copy / f.name).write_bytes(f.read_bytes())
    monkeypatch.setattr(bench, "ROOT", tmp_path)
    seen = {bench.pass_sources_digest()}
    for name in sorted(files):
        with (copy / name).open("a") as f:
            f.write("\n// changed\n")
        seen.add(bench.pass_sources_digest())
    assert len(seen) == 1 + len(files)
