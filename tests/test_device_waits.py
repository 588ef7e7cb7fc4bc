"""What the device-side waits have to keep to, read off the CUDA sources (no GPU needed): a time-out cannot be produced in
the product kernels without holding up a GPU, so the rules that make it end are checked where they are written."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_06183_b200", "csrc")


def _sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def test_roles_of_whole_warps_wait_as_a_warp():
    """Accumulators, packed tiles and scored strips are consumed by whole warps (aligned TMEM loads, shuffles, named
    barriers): these waits give one answer to the warp. A wait answered lane by lane would let lanes part at an expiry."""
    collective = re.compile(r"\bmbar_wait\(\s*(?:&ctl->(?:tmem_full|pk_full|scored)\b|tmem_full_bar\b)")
    for name, text in _sources().items():
        assert not collective.search(text), name
    stream = _sources()["vnm_stream.cu"]
    assert not re.search(r"\bmbar_wait\(&ctl->full\b", stream)          # scoring warps: shuffles and named barriers


def test_warps_that_meet_at_named_barriers_leave_together():
    """A warp that gave up must not leave the others of its set waiting at a named barrier: the sets that use one vote."""
    assert re.search(r"named_all\(set \+ 1, 128, ok\)", _sources()["gemm_tc.cu"])
    assert re.search(r"if \(!named_all\(1, 128, ok\)\) break;", _sources()["vnm_stream.cu"])


def test_kernels_with_copies_in_flight_drain_them_after_an_expired_wait():
    """A CTA that leaves early must not hand its shared memory on while copies into it are under way."""
    kernels = 0
    for name, text in _sources().items():
        for body in re.split(r"\n__global__ ", text)[1:]:
            body = body[:body.index("\n}\n")]
            if re.search(r"\b(tma_load_2d|tma_load_2d_2cta|bulk_load|tma_gather4_2d)\(", body):
                kernels += 1
                assert "drain_after_expiry()" in body, (name, body[:200])
    assert kernels == 6          # three products, two streaming sparsifiers, the strided prune


def test_kernels_that_take_all_of_tmem_have_an_sm_to_themselves():
    """Every launcher of a kernel that allocates tensor memory asserts at compile time that two such CTAs do not fit one SM:
    a CTA placed beside its predecessor's would sit in the allocation, which has no time limit."""
    text = _sources()["gemm_tc.cu"]
    allocating = [b for b in re.split(r"\n__global__ ", text)[1:] if "tmem_alloc" in b[:b.index("\n}\n")]]
    assert len(allocating) == 3
    assert len(re.findall(r"static_assert\(.*kExclusiveSmem", text)) == 3          # one-CTA, CTA-pair and 512-row kernels
