"""Rules of the CUDA sources that a run cannot show to be broken (it works until
the scheduling changes), checked by reading the kernels on CPU."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_31035_gb300", "csrc")


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def kernels():
    """(file, name, parameters, body) of every __global__ function."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        text = strip_comments(open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\(([^{]*)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out.append((f, m.group(1), m.group(2), text[m.end():i]))
    return out


KERNELS = kernels()


def test_every_kernel_is_found():
    launches = sum(len(re.findall(r"__global__", strip_comments(open(os.path.join(CSRC, f)).read())))
                   for f in os.listdir(CSRC))
    assert len(KERNELS) == launches > 20


# CUDA defines accesses to another CTA's shared memory only once that CTA has
# started, which a barrier of the whole cluster is the way to know.
REMOTE = [k for k in KERNELS if re.search(r"mapa_shared|st_cluster", k[3])]


@pytest.mark.parametrize("name,body", [(k[1], k[3]) for k in REMOTE], ids=[k[1] for k in REMOTE])
def test_cluster_barrier_before_remote_shared_memory(name, body):
    barrier = re.search(r"\bcluster_(sync|wait)\s*\(\s*\)", body)
    remote = re.search(r"\bst_cluster_\w+\s*\(|\bmbar_arrive_cluster\s*\(|\bmma_commit_pair\s*\(", body)
    assert barrier and remote and barrier.start() < remote.start(), name


# A programmatic dependent runs while the kernel before it still writes, so
# nothing it reads may go through the non-coherent path, whose data must be
# constant for the whole kernel and whose loads may be moved above the wait.
DEPENDENT = [k for k in KERNELS if "griddep_wait" in k[3]]


@pytest.mark.parametrize("params,body", [k[2:] for k in DEPENDENT], ids=[k[1] for k in DEPENDENT])
def test_dependents_read_coherently(params, body):
    assert not re.search(r"__ld(g|cg|ca|cs|lu)\s*\(", body)
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params)


def test_shared_device_code_reads_coherently():
    for f in sorted(os.listdir(CSRC)):
        text = strip_comments(open(os.path.join(CSRC, f)).read())
        assert "ld.global.nc" not in text, f
        if f.endswith(".cuh"):
            assert "__ldg" not in text, f


# The status bits that the header documents: 1 a producer's wait, 2 / 4 the
# MMA thread's for an accumulator or a stage, 8 its final drain.
PIPELINED = [k for k in KERNELS if "fail(" in k[3]]


@pytest.mark.parametrize("body", [k[3] for k in PIPELINED], ids=[k[1] for k in PIPELINED])
def test_status_bits_name_their_role(body):
    roles = re.split(r"(?:else )?if \(warp\b", body)[1:]
    mma = [bool(re.search(r"\bmma_(f16|nvf4)\w*\s*\(", r)) for r in roles]
    assert any(mma)
    for r, issues_mma in zip(roles, mma):
        bits = set(re.findall(r"fail\((\d+)u\)", r))
        assert issues_mma or not bits & {"2", "4", "8"}
        if "tma_load_2d" in r and not issues_mma:
            assert bits <= {"1"}


@pytest.mark.parametrize("body", [k[3] for k in KERNELS], ids=[k[1] for k in KERNELS])
def test_flat_indices_hold_the_largest_sizes(body):
    """A flat index over all threads is not a signed 32-bit number: 64 rows of
    K = 2^30, which the GEMMs take, are 2^31 chunks of 32."""
    assert not re.search(r"\bint\s+\w+\s*=\s*(\(int\)\s*)?\(?\s*blockIdx\.x\s*\*", body)
