"""Orderings and sizes in the source (csrc) that no run can be relied on to show."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNELS = os.path.join(ROOT, "paper_1101_0423_gb300", "csrc", "dwf_kernels.cuh")


def test_refilled_link_buffer_is_fenced_against_its_staging_rows():
    """k_hop with one link buffer stages results in the buffer's bytes with ordinary stores and
    then, when a CTA walks several tiles, refills it by bulk copies.  Those write through the
    async proxy: every thread's fence.proxy.async has to stand before the barrier that precedes
    the copy, or a late store may land in the new links."""
    src = re.sub(r"//[^\n]*", "", open(KERNELS).read())
    assert re.search(r"void fence_proxy_async\(\)\s*\{\s*asm volatile\(\"fence\.proxy\.async\.shared::cta;\"", src)
    loop = src[src.index("for (long tile = blockIdx.x"):]
    refill = loop.index("issue(tile, 0)")
    before = re.sub(r"\s+", " ", loop[:refill])
    assert re.search(r"if \(it > 0\) \{ fence_proxy_async\(\); __syncthreads\(\); if \(tid == 0\) \{", before)
    # no other bulk copy reuses bytes that ordinary stores wrote: the first copy of a CTA and
    # the double-buffered ones, whose buffers are only read
    assert loop.count("issue(") == 2 and src.count("issue(") == 3


def test_server_counts_the_links_as_the_kernels_store_them():
    """The server's budget takes a gauge ensemble's bytes from the link layouts' own constants, so
    that a padded site is counted with its padding."""
    src = open(os.path.join(os.path.dirname(KERNELS), "dwf_server.cu")).read()
    body = re.search(r"size_t gauge_bytes\(.*?\n}\n", src, re.S).group()
    assert [p in body for p in ("PT<P_F64>::SITE_LREALS * 8", "PT<P_F32>::SITE_LREALS * 4", "PT<P_F16>::SITE_LREALS * 2")] == [True] * 3
    assert not re.search(r"\b(1152|656|192)\b", body)
