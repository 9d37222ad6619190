"""Rules that every kernel of the library keeps because all of them are launched with programmatic stream serialisation,
checked on the sources (what they prevent is a race: it shows on a device now and then or never)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_19705_b200", "csrc")


def _strip(text):
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


def _close(text, i, pair):
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == pair[0]) - (text[j] == pair[1])
        if depth == 0:
            return j
    raise ValueError("unbalanced source")


def _functions(marker):
    """(file, name, body) of every function defined after `marker`."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = _strip(open(path).read())
        for m in re.finditer(marker, text):
            head = re.compile(r"(\w+)\s*\(").search(text, m.end())
            while head.group(1) in ("__launch_bounds__", "__align__"):
                head = re.compile(r"(\w+)\s*\(").search(text, _close(text, head.end() - 1, "()") + 1)
            end = _close(text, head.end() - 1, "()")
            if text[end + 1:].lstrip()[:1] != "{":
                continue  # a declaration
            body = text.index("{", end)
            out.append((os.path.basename(path), head.group(1), text[body + 1:_close(text, body, "{}")].strip()))
    return out


KERNELS = _functions(r"__global__")


def test_kernels_are_found():
    assert len(KERNELS) > 60 and {"ns_block_kernel", "bd_pass_kernel", "wait_probe_kernel"} <= {n for _, n, _ in KERNELS}


@pytest.mark.parametrize("file,name,body", KERNELS, ids=[f"{f}-{n}" for f, n, _ in KERNELS])
def test_kernel_waits_for_its_predecessor_first(file, name, body):
    assert re.match(r"pdl_(enter|wait)\(\);", body), f"{name} does not begin with the wait for the kernel before it"


# functions that meet at a barrier or exchange values between lanes, directly or in what they call
COLLECTIVE = re.compile(r"__syncthreads|__syncwarp|_sync\(|mbar_|block_sum_double|gauss_jordan|pw_norm2")


@pytest.mark.parametrize("file,name,body", [f for f in KERNELS + _functions(r"__device__ __forceinline__ void(?= bd_)") if COLLECTIVE.search(f[2])],
                         ids=lambda v: v if isinstance(v, str) and len(v) < 40 else "")
def test_a_block_stops_as_a_whole(file, name, body):
    """The status word may be raised while a block starts.  Threads that looked at it one by one could disagree, and those
    that went on would wait at barriers for the ones that left."""
    assert not re.search(r"if \([^;{]*\*\s*(\w+\.)?status\)", body), f"{name}: every thread reads the status word for itself"


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_inputs_are_read_with_ordinary_loads(path):
    """An overlapped kernel's inputs change during its lifetime: no read-only loads, and no promise that allows them."""
    text = _strip(open(path).read())
    assert not re.search(r"__ldg\b|ld\.global\.nc", text)
    assert not re.search(r"\bconst\s+\w+\s*\*\s*__restrict__", text)


RETURNING = (r"launch_dense_tc6?|launch_kk_tc|tg_launch|tb_launch|bd_launch\w*|bw_launch\w*|ns_block_launch|kk_chain_launch|ns_inverse|"
             r"minv_path_tc|penalty_tc|opgrad_\w+_tc|pinv_rows|dense_product|dense_pqe|alg1_run")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_launch_result_is_dropped(path):
    """A launch that could not be made (an operand that a tensor map does not take) must end the call, not leave stale results."""
    dropped = re.findall(r"[;{})]\s*((?:%s)\s*\([^;{}]*;)" % RETURNING, _strip(open(path).read()))
    assert not dropped, dropped
    assert not re.search(r"static void (%s)\(" % RETURNING, _strip(open(path).read()))


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_launch_result_of_a_paired_product_is_dropped(path):
    names = r"launch_split_product|tg_launch_\w+|t2_launch|pinv_loop_launch|gram_inverse"
    text = _strip(open(path).read())
    assert not re.findall(r"[;{})]\s*((?:%s)\s*\([^;{}]*;)" % names, text)
    assert not re.search(r"static void (%s)\(" % names, text)


def _enclosing(text, pos):
    """Heads of the blocks that the position lies in, the innermost first."""
    heads, depth = [], 0
    for j in range(pos - 1, -1, -1):
        if text[j] == "}":
            depth += 1
        elif text[j] == "{":
            if depth == 0:
                heads.append(re.split(r"[;{}]", text[:j])[-1].strip())
            else:
                depth -= 1
    return heads


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_named_barriers_do_not_depend_on_a_wait(path):
    """A bounded wait may give up in one warp and succeed in another; a barrier that only the second reaches has no limit."""
    text = _strip(open(path).read())
    for m in re.finditer(r"bar\.sync|barrier\.sync", text):
        assert not [h for h in _enclosing(text, m.start()) if re.match(r"(else )?if \(.*\b(ok|mbar_wait)\b", h)]


def test_operands_for_the_other_cta_are_released_at_cluster_scope():
    """The issuing CTA of a pair multiplies what the other CTA's builders stored: what arrives there on their behalf, and its wait, order
    those stores for it only at the scope of the cluster.  The builders themselves arrive in their own CTA, where a relay waits."""
    text = _strip(open(os.path.join(CSRC, "kernels_bwd.cuh")).read())
    body = text[text.index("void bd_bwd_pair_body"):text.index("constexpr int bw_threads")]
    assert re.findall(r"(mbar_\w+)\(sfull0", body) == ["mbar_arrive_pair"]
    assert sorted(re.findall(r"(mbar_wait\w*|wait_all)\(bar_sfull", body)) == ["mbar_wait", "mbar_wait_pair"]
    assert re.findall(r"(mbar_arrive\w*)\(bar_sfull", body) == ["mbar_arrive"]
    pair = _strip(open(os.path.join(CSRC, "kernels_pair_mma.cuh")).read())
    assert "mbarrier.arrive.release.cluster.shared::cluster" in pair and "try_wait.parity.acquire.cluster" in pair
