"""The traffic table trusts a capture while the hash of the kernel's sources holds,
so the hashed list has to hold every file of csrc that those sources include;
and the kernel of a one-launch step is found without being named."""
import json
import os
import re

import pytest

from paper_1505_02037_gb300 import traffic_table as TT

CSRC = os.path.join(os.path.dirname(TT.__file__), "csrc")


@pytest.mark.parametrize("name", ["COLLIDE_SOURCES", "AD_SOURCES", "BATCH_SOURCES"])
def test_every_included_source_is_hashed(name):
    listed = set(getattr(TT, name))
    for f in listed:
        with open(os.path.join(CSRC, f)) as fh:
            for inc in re.findall(r'#include "([^"]+)"', fh.read()):
                if not inc.startswith(".."):  # the public header declares no kernel
                    assert inc in listed, (f, inc)


def test_one_launch_kernel_is_found(tmp_path):
    cap = tmp_path / "cap.csv"
    rows = [(0, "void k_init<19>(...)", "dram__bytes_read.sum", "byte", "7"),
            (1, "void k_step<19>(...)", "dram__bytes_read.sum", "byte", "13000"),
            (1, "void k_step<19>(...)", "dram__bytes_write.sum", "byte", "12000")]
    head = '"ID","Kernel Name","Metric Name","Metric Unit","Metric Value"\n'
    cap.write_text(head + "".join('"%d","%s","%s","%s","%s"\n' % r for r in rows))
    out = tmp_path / "table.json"
    assert TT.main([str(cap), "--key", "k", "--cells", "10", "--out", str(out), "--captured-on", "t",
                    "--command", "ncu"]) == 0
    assert json.loads(out.read_text())["k"]["dram_bytes_per_cell"] == 2500.0
