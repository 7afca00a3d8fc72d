"""What orders the accesses of a cluster's CTAs, and of a CTA's roles, in the 64-bit kernels, read from the source.

A missing barrier shows in a run only when one CTA falls behind another in a window of a few hundred cycles, so
these tests check that the ordering statement is where the shared memory is reused.
"""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_14741_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())  # without comments


def body(text, name):
    """The text of the function `name`, from its opening brace to the matching one."""
    for m in re.finditer(r"\b%s\(" % name, text):  # (its definition: followed by a brace)
        i, depth = m.end(), 1
        while depth:  # past the parameters
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if text[i:].lstrip().startswith("{"):
            start = i = text.index("{", i)
            while True:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
                if not depth:
                    return text[start:i]
    raise AssertionError(f"no function {name}")


def test_bound_exchange_is_read_before_its_memory_is_reused():
    # the exchanged row sums lie where the caller's next pass writes digits: every CTA's last read of them comes
    # before a barrier of the cluster
    b = body(source("k_ns_fp64.cu"), "first_bound")
    last = b.rindex("share(")
    assert "phase_sync()" in b[last:]


def test_column_norms_are_read_before_the_matrix_changes():
    # the maximum over the cluster's CTAs ends in a barrier, so the callers may change the matrix in place
    text = source("k_ns_fp64.cu")
    assert "cluster_max(" in body(text, "column_norm2") and "phase_sync()" in body(source("smx_slices.cuh"), "cluster_max")


def test_row_lengths_are_read_before_they_are_cleared():
    # the coupled iteration's sums: added to in a pass, read after its barrier, cleared after one more barrier
    b = body(source("k_ns_fp64.cu"), "coupled_steps")
    b = b[b.index("for (int it"):]
    at = [b.index(x) for x in ("clear_sums(row_y, 2 * k)", "pass_residual(", "longest(row_r)", "slice_product(sh, jb.P[0], jb.P[2]", "clear_sums(row_r, k)",
                               "pass_update(Y", "slice_product(sh, jb.P[2], jb.P[1]", "pass_update(Z", "longest(row_z)", "longest(row_y)",
                               "pass_affine(Z, shift ? Z")]
    assert at == sorted(at)


def test_a_claimed_job_is_read_before_its_word_is_written_again():
    # between two claims there may be no barrier of the cluster: two words in turn, so that the write of one is
    # ordered after its last read by the claim between them
    b = body(source("k_ns_fp64.cu"), "claim_job")
    word = re.search(r"(\w+) \+ \(round & 1\)", b)
    assert word and b.index(word.group(0)) < b.index("__stcg(") < b.index("phase_sync()") < b.index("__ldcg(")


def test_readers_of_an_accumulation_give_up_together():
    # the 14 reading warps meet at barrier 1 once per accumulation: one decision, published before the barrier
    b = body(source("smx_slices.cuh"), "slice_product")
    readers = b[b.index("bar.sync 1, 448") - 300:]
    assert readers.index("sh->gave_up[use & 1] = *ab") < readers.index("bar.sync 1, 448")
    after = readers[readers.index("bar.sync 1, 448"):]
    assert after.index("alive = !sh->gave_up[use & 1]") < after.index("++use")
    assert "*ab" not in after  # no warp looks at the flag for itself


def test_bound_vectors_leave_the_stage_area_before_it_ends():
    # two vectors of 64-bit words per row in shared memory; past a size they lie in the slot
    text, slices = source("k_ns_fp64.cu"), source("smx_slices.cuh")
    rows = int(re.search(r"kBoundSharedRows = (\d+)", text).group(1))
    planes, tile, stages = (int(re.search(r"%s = (\d+)" % c, slices).group(1)) for c in ("kSlicePlanes", "kSliceTile", "kSliceStages"))
    assert 16 * rows <= stages * planes * 32 * (128 + tile)
    assert "k <= kBoundSharedRows ?" in body(text, "first_bound")


def test_dense_entry_point_keeps_a_pending_error():
    # the runtime's last error is the caller's: it is not read (which clears it), and a launch is tried once, with a
    # cluster that the device has been asked about
    text = source("k_ns_fp64.cu")
    b = body(text, "smx_dense_density_noalloc")
    assert "cudaGetLastError" not in b and b.count("launch_clusters(") == 1 and "kernel_clusters(" in b
    assert "cudaGetLastError" not in body(source("k_ns_graded.cu"), "launch_dense_graded")
