"""What a kernel's role hands to another through shared memory is stored before
the arrival that releases it.  A store after the arrival is a race that the
latency of a copy or of a cluster hides from every run, so the order is checked
in the source."""
import os

from paper_2607_20791_gb300.build import CSRC


def _between(name, start, end):
    text = open(os.path.join(CSRC, name)).read()
    at = text.index(start)
    return text[at:text.index(end, at)]


def test_page_descriptors_precede_the_k_arrival():
    # the softmax reads descs after s_full, whose arrival by the QK thread follows its wait on k_full
    role = _between("attention_kernel.cuh", "if (valid && gidx == gq) {", "atomicMax(&s_issued")
    store, arrive = role.index("descs["), role.index("mbar_arrive_expect_tx(&full[gs]")
    assert store < arrive
    assert "descs[" not in role[arrive:]


def test_row_flags_are_read_before_the_row_parameters_arrive():
    # a stream warp's maximum waits for its draw warp's arrival on prm_bar; a finished row's
    # flag may be cleared behind the exchange of the maxima, so a draw warp that read the
    # block's flags after its arrival could miss an active row
    role = _between("sample_head.cu", "draw warp ====", "no CTA leaves while another")
    arrive = role.index("mbar_arrive(&sh.prm_bar")
    assert role.index("p.row_active[row]") < role.index("__ballot_sync") < arrive
    assert "row_active" not in role[arrive:] and "block_rows" not in role
