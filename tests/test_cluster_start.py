"""Every cluster kernel passes a cluster barrier before it first writes another
CTA's shared memory (CUDA gives access to a CTA's shared memory only once that
CTA has started).  A launch may not show a missing one, so the sources are read:
in the body of a kernel with __cluster_dims__, outside lambdas, the first
cluster.sync() stands before the first call or store that writes to a peer."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_04323_gb300", "csrc")


def braces(src, at):
    """The text of the block whose opening brace is the first one at or after `at`, and its end."""
    start, depth = src.index("{", at), 0
    for i in range(start, len(src)):
        depth += (src[i] == "{") - (src[i] == "}")
        if depth == 0:
            return src[start:i + 1], i + 1
    raise AssertionError("unbalanced braces")


def cluster_kernels():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            for m in re.finditer(r"__cluster_dims__\([^)]*\)[^{;]*?(\w+)\s*\(const", src):
                yield name, m.group(1), braces(src, m.end())[0]


def first_barrier_and_write(body):
    """Offsets of the first cluster barrier and of the first write to a peer, by a
    store through map_shared_rank or a peer pointer, or by a lambda that holds one."""
    writers = []
    plain = body
    for m in re.finditer(r"auto (\w+) = \[&\]", body):
        text, end = braces(body, m.end())
        if re.search(r"peer\[|map_shared_rank", text):
            writers.append(m.group(1))
        plain = plain[:m.start()] + " " * (end - m.start()) + plain[end:]  # offsets stay
    write = re.compile(r"map_shared_rank\([^;]*?\)\[[^;]*\] =[^=]|peer\[[^;=]*\]\[[^;]*\] =[^=]"
                       + "".join(rf"|\b{w}\(" for w in writers))
    found = write.search(plain)
    return plain.find("cluster.sync()"), found.start() if found else None


def test_barrier_before_the_first_write_to_a_peer():
    seen = []
    for name, kernel, body in cluster_kernels():
        barrier, write = first_barrier_and_write(body)
        assert write is not None, f"{name} {kernel}: no write found"
        assert 0 <= barrier < write, f"{name} {kernel}: writes to a peer before the cluster's first barrier"
        seen.append(kernel)
    assert len(seen) >= 2, seen
