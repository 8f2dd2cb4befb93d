"""Order of shared-memory accesses in the kernels that stage bulk copies, read from their source: what a
run cannot show, since the wrong order gives wrong results only now and then."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc")
KERNELS = [("k_rows.cuh", "row_fwd_kernel"), ("k_rows.cuh", "row_anom_kernel"), ("k_rows.cuh", "row_inv_kernel"),
           ("k_cols.cuh", "col_stats_kernel"), ("k_cols.cuh", "col_update_kernel")]


def _body(file, kernel):
    """The kernel's body without comments."""
    with open(os.path.join(CSRC, file), encoding="utf-8") as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    at = text.index("{", re.search(r"\b%s\(const" % kernel, text).end())
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            return text[at:end]


@pytest.mark.parametrize("file,kernel", KERNELS)
def test_verdict_is_read_before_the_word_is_written_again(file, kernel):
    """cta_wait leaves its verdict in a shared word that every thread reads after a CTA barrier; the next wait
    with the same word needs another CTA barrier first (line barriers do not hold the whole CTA)."""
    body = _body(file, kernel)
    waits = [(m.end(), m.group(1)) for m in re.finditer(r"cta_wait\(.*?p\.status, (\w+)(?:, expire)?\)", body)]
    assert waits
    for n, (end, word) in enumerate(waits):
        later = [w for w in waits[n + 1:] if w[1] == word]
        until = later[0][0] if later else len(body)   # the word's next wait, or its own in the next pass of the loop
        assert "__syncthreads()" in body[end:until], word


@pytest.mark.parametrize("file,kernel", KERNELS + [("k_colf.cuh", "col_fused_kernel")])
def test_stage_is_fenced_before_its_next_copy(file, kernel):
    """In the loop over the staged units, every barrier after which one thread issues a copy into a stage is
    preceded by the fence that orders the threads' accesses to that stage before the copy, with no other barrier
    in between.  (issue_w of the column update follows a later barrier: its stage is read before the gain stage,
    whose fence covers both.)"""
    body = _body(file, kernel)
    barrier = r"__syncthreads\(\)|line_sync<T>\(bid\)|cta_wait\("
    loop = re.search(r"for \([^;]*; (q < Q|cb < ncol|base < n_items|c < ncol)", body).start()   # past the first copies
    issues = [m.start() for m in re.finditer(r"issue(?:_next|_tile|_rows|_g)?\(", body) if m.start() > loop]
    assert issues
    for at in issues:
        barriers = [m.start() for m in re.finditer(barrier, body[:at])]
        assert "stage_reads_done()" in body[barriers[-2]:barriers[-1]], body[at:at + 40]
