"""No copy or commit of the library is multicast over a cluster: it runs on machines with
several GPUs (partitioned batches), where such loads are not used."""
import glob
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_07551_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*"))))
def test_source_has_no_cluster_multicast(name):
    with open(os.path.join(CSRC, name)) as f:
        assert ".multicast" not in f.read()
