"""Kernels that store into or load from another CTA's shared memory first wait on a cluster barrier.

A CTA of a cluster may run before another one of it has started, and an access to the shared memory of a CTA
that has not started is undefined. The sources are read as text: in every kernel (and in the device functions
before a file's first kernel) the first remote access follows a wait on the cluster barrier.
"""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2511_09844_gb300", "csrc")
REMOTE = re.compile(r'\b(st_dsmem\w*|st_async\w*|ld_dsmem\w*)\s*\(|"st\.shared::cluster')
WAIT = re.compile(r"\b(cluster_sync_all|cluster_wait)\s*\(\)")


def _parts(path):
    """The file's code from kernel to kernel, without comments and without the one-line wrappers' heads."""
    text = re.sub(r"//[^\n]*", "", open(path).read())
    text = "\n".join(ln for ln in text.split("\n") if not ln.lstrip().startswith("__device__"))
    return text.split("__global__")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_remote_accesses_follow_a_cluster_wait(name):
    for part in _parts(os.path.join(CSRC, name)):
        remote = REMOTE.search(part)
        if not remote:
            continue
        wait = WAIT.search(part)
        assert wait and wait.start() < remote.start(), part[max(0, remote.start() - 200):remote.end()]
