"""The key under which a recorded DRAM traffic figure is valid covers all that the kernel is made of."""
import os
import shutil

import bench


def test_traffic_key_covers_the_included_files(tmp_path):
    csrc = tmp_path / "csrc"
    shutil.copytree(os.path.join(bench.ROOT, "paper_2209_04487_gb300", "csrc"), csrc)
    first = {k: bench._source_digest(str(csrc / k)) for k in ("mol_rotor.cu", "mol_col.cu")}
    assert first == {k: bench._source_digest(os.path.join(bench.ROOT, "paper_2209_04487_gb300", "csrc", k))
                     for k in first}
    for header, used in (("mol_fft.cuh", {"mol_rotor.cu"}), ("mol_common.cuh", set(first)),
                         ("ms_internal.cuh", set(first)), ("yee.cu", set())):
        text = (csrc / header).read_text()
        (csrc / header).write_text(text + "\n")
        assert {k for k in first if bench._source_digest(str(csrc / k)) != first[k]} == used
        (csrc / header).write_text(text)
