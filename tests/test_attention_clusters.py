"""How many clusters are resident is kept per kernel: the attention's four kernels
(d x query rows of a tile) differ in shared memory, and the count sets the plan, so
no kernel may take the count of the one that ran first."""
import re
import shutil
import subprocess

import pytest


def test_one_table_of_resident_clusters_per_kernel():
    if shutil.which("nm") is None:
        pytest.skip("needs nm")
    from paper_2606_20543_gb300 import build
    names = subprocess.run(["nm", "-C", build.build()], capture_output=True, text=True,
                           check=True).stdout
    tables = {m for m in re.findall(r"resident_clusters<([^>]*)>\(\)::known", names)}
    assert tables == {"64, 64", "64, 128", "128, 64", "128, 128"}
