"""The bench reports a captured traffic figure only while every source that the attention
kernels are compiled from is the one it was captured with."""
import os
import shutil

import pytest

import bench
from paper_2609_34538_gb300.build import CSRC


def test_every_included_file_counts():
    for f in bench.ATTENTION_SOURCES:
        for line in open(os.path.join(CSRC, f)):
            if line.startswith('#include "') and f.startswith("das_"):
                name = line.split('"')[1]
                assert name in bench.ATTENTION_SOURCES or name == "das.h", f"{f} includes {name}"


@pytest.mark.parametrize("name", bench.ATTENTION_SOURCES)
def test_an_edit_of_any_source_changes_the_digest(name, tmp_path):
    for f in bench.ATTENTION_SOURCES:
        shutil.copy(os.path.join(CSRC, f), tmp_path)
    before = bench.attention_digest(tmp_path)
    path = tmp_path / name
    text = path.read_text()
    path.write_text("// a comment\n" + text)
    assert bench.attention_digest(tmp_path) == before
    path.write_text(text + "int edited;\n")
    assert bench.attention_digest(tmp_path) != before
