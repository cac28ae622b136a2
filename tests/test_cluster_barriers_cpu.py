"""Distributed shared memory may only be touched once every CTA of the cluster is known to have started.
What a kernel does before that cannot be provoked on purpose, so it is read in the sources: in every
function, a cluster barrier stands in front of the first access to another CTA's shared memory, and
another one behind the last, before that CTA may have left."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_15023_b200", "csrc")
BARRIER = re.compile(r"barrier\.cluster\.wait|this_cluster\(\)\.sync\(\)|\bcluster\.sync\(\)")


def _functions(text):
    """Bodies of the functions of a file: the outermost braces inside namespaces."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"(extern \"C\"|namespace( \w+)?)\s*\{", "", text)
    depth = start = 0
    for m in re.finditer(r"[{}]", text):
        if m.group() == "{":
            if depth == 0:
                start = m.start()
            depth += 1
        elif depth:
            depth -= 1
            if depth == 0:
                yield text[start:m.end()]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_remote_shared_memory_stands_between_cluster_barriers(path):
    for body in _functions(open(path).read()):
        remote = [m.start() for m in re.finditer(r"map_shared_rank", body)]
        if remote:
            barriers = [m.start() for m in BARRIER.finditer(body)]
            assert barriers and min(barriers) < min(remote), body[:200]
            assert max(barriers) > max(remote), body[:200]
