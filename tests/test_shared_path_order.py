"""Order of the strain path's shared-memory accesses in the source (CPU): the path is read by
volatile inline assembly without a memory clobber, which a compiler may move across ordinary
stores, so the only stores to it stand between two compiler barriers."""
import re
from pathlib import Path

SRC = Path(__file__).resolve().parent.parent / "paper_2402_09996_gb300" / "csrc" / "constitutive.cuh"


def test_path_stores_stand_between_compiler_barriers():
    text = re.sub(r"//[^\n]*", "", SRC.read_text())
    assert "ld.shared" in text
    body = re.search(r"void store_path\(.*?\{(.*?)\n\}", text, re.S)
    assert body, "the path has one writer"
    barrier = 'asm volatile("" ::: "memory")'
    parts = [p.strip() for p in body.group(1).split(";") if p.strip()]
    stores = [k for k, p in enumerate(parts) if p.startswith("d[")]
    assert stores and barrier in parts[: stores[0]] and barrier in parts[stores[-1] + 1 :]
    # no other store to the path's buffer
    assert len(re.findall(r"reinterpret_cast<float4\*>\(sc\)", text)) == 1
