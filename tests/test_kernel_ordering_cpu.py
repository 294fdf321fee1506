"""Memory-ordering rules of the one-kernel compressors, checked on their source text (no GPU run can show that an order is
guaranteed): every word that other CTAs wait for is published with release where the readers rely on other stores."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_03298_b200", "csrc")

# words whose readers use nothing but the word (the parameters of the sample, a count of blocks, and the parameters of the whole
# tensor as long as nothing is written on the strength of them: a second pass waits for all_left)
STANDS_FOR_ITSELF = {"ctl->params[0]", "ctl->pack_target", "ctl->verdict"}


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_words_that_order_stores_are_published_with_release():
    text = _source("enec_fused.cuh") + _source("enec_fused_list.cuh")
    awaited = set(re.findall(r"await_published\(&([\w>\[\].-]+)", text))
    assert awaited == {"ctl->params[which]", "ctl->pack_target", "ctl->verdict", "ctl->all_left", "ctl.ready"}
    relaxed = set(re.findall(r"publish_word\(&([\w>\[\].-]+)", text))
    released = set(re.findall(r"\bpublish\(&([\w>\[\].-]+)", text))
    assert relaxed <= STANDS_FOR_ITSELF, relaxed - STANDS_FOR_ITSELF
    assert {"ctl->params[1]", "ctl->all_left", "ctl.ready"} <= released
    assert "st.release.gpu" in re.search(r"void publish\(.*?\n}", text, re.S).group(0)


def test_other_lanes_read_behind_a_barrier_after_one_lane_acquires():
    """A shuffle passes a value on, it orders no memory access: between one lane's acquire and the others' reads stands a
    __syncwarp()."""
    scout = re.search(r"auto scout_middle = .*?\n    };", _source("enec_fused_list.cuh"), re.S).group(0)
    counted = re.search(r"void first_pass_counted\(.*?\n}", _source("enec_fused.cuh"), re.S).group(0)
    assert scout.index("ld.acquire") < scout.index("__syncwarp()") < scout.index("ld_relaxed_u32(from")
    assert counted.index("add_acq_rel(") < counted.index("__syncwarp()") < counted.index("search_global")


def test_the_loss_flag_is_read_behind_a_fence_of_every_lane():
    """The lanes that look up the last block's offset read other CTAs' counts; the flag that those CTAs set before is read after a
    fence by each of these lanes and a barrier, and before the header is written."""
    text = _source("enec_fused.cuh")
    finish = re.search(r"void finish_block\(.*?\n}", text, re.S).group(0)
    order = [finish.index(s) for s in ("__threadfence()", "__syncwarp()", "(threadIdx.x & 31) != 0", "t.lossy", "Header hd;")]
    assert order == sorted(order)
    say = re.search(r"auto say_lossy = .*?\n    };", text, re.S).group(0)
    assert say.index("leave_no_stream(t)") < say.index("&ctl->lossy") < say.index("__threadfence()")


def test_a_wait_that_ran_out_leaves_no_stream():
    """No run makes these bounded waits end early, so their error paths are read here: wherever one reports ENEC_ERR_TIMEOUT, the
    header's magic and the length are zeroed too (the output may hold an earlier stream), and a block whose records were
    not placed takes its count back, so that the last block's CTA does not write a header."""
    text = _source("enec_fused.cuh")
    give_up = re.search(r"void give_up\(.*?\n}", text, re.S).group(0)
    for part in ("report(status, ENEC_ERR_TIMEOUT)", "t.state[k], 0ull", "&t.super[k / kSuperBlocks]", "leave_no_stream(t)"):
        assert part in give_up
    rest = text.replace(give_up, "")
    assert len(re.findall(r"if \(!sh\.ok\) (?:{ )?lost = ", rest)) == 2     # waiting block, block without room to wait
    assert rest.count("if (lost && tid == 0) give_up<DT>(lost, status);") == 1
    for report in re.finditer(r"report\(status, ENEC_ERR_TIMEOUT\);", rest):
        assert re.match(r"\s*leave_no_stream\(t\);", rest[report.end():])
    text = _source("enec_fused_list.cuh")
    assert len(re.findall(r"lost = (?:pend_)?slot << 28", text)) == 3       # those two, and a CTA that waits for parameters
    end = text[text.index("if (stop) {"):]
    assert text.count("report(status, ENEC_ERR_TIMEOUT)") == end.count("report(status, ENEC_ERR_TIMEOUT)") == 1
    assert "give_up<DT>(" in end and "i < list.n_items" in end and "->magic = 0" in end and "out_size = 0" in end
    assert not re.search(r"\breturn;", text[text.index("enec_fused_list_kernel("):text.index("if (stop) {")].split("for (uint32_t iter = 0;;")[1])
