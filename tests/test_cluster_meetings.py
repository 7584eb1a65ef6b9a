"""A CTA may write into another CTA's shared memory only once that CTA has started, so every kernel that maps a peer's
shared memory has to wait for its cluster before it does. Read off the sources: the race cannot be provoked."""
import glob
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2312_05693_b200", "csrc")
WAIT = re.compile(r"barrier\.cluster\.wait|cluster_started_wait\(\)|cluster_meet\(\)|cluster\.sync\(\)")


REMOTE = re.compile(r"map_shared_rank|leave_range\b")           # leave_range stores through a pointer that its caller has mapped


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for part in open(path).read().split("__global__")[1:]:
            part = re.sub(r"//[^\n]*", "", part)
            if REMOTE.search(part):
                yield pytest.param(part, id=re.search(r"(\w+_kernel)\(", part).group(1))


@pytest.mark.parametrize("body", list(kernels()))
def test_remote_stores_come_behind_a_wait_for_the_cluster(body):
    first = REMOTE.search(body).start()
    helper = re.search(r"auto (\w+) = \[&\]\([^)]*\) \{[^{}]*map_shared_rank", body)     # a store inside a lambda counts where it is called
    if helper:
        first = body.index(helper.group(1) + "(", helper.end())
    assert WAIT.search(body, 0, first), "stores into a peer's shared memory before the cluster is known to have started"


def test_the_headers_map_no_peer_themselves():
    """What the headers hold is not read as part of a kernel above: the only store into a peer there goes through a pointer that
    the kernel hands in."""
    stores = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert "map_shared_rank" not in code and "mapa" not in code, path
        stores += re.findall(r"\*\s*(peer_\w+)\s*=", code)
    assert stores == ["peer_slot"]
    users = [k.id for k in kernels() if "leave_range" in k.values[0]]
    assert sorted(users) == ["log2_absmax_kernel", "range_kernel"]


def test_asynchronous_remote_stores_come_behind_it_too():
    """Kernels that send to a peer by st.async map its memory with mapa: behind a wait for the cluster in the same function, and
    (the stores at the end of the few-row kernel) in the kernel's own text before them."""
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for at in (m.start() for m in re.finditer(r'"mapa\.', code)):
            body = code[max(code.rfind("\n}\n", 0, at), 0):at]
            assert WAIT.search(body), path
            found += 1
    assert found >= 6


def test_waits_for_what_peers_send_are_at_their_scope():
    """A barrier that other CTAs' st.async count on (its address goes through mapa) is waited for at the scope of the cluster:
    without a scope the wait orders nothing that another CTA wrote."""
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        mapped = set(re.findall(r'"mapa\.[^;]*;" : "=r"\(bar\) : "r"\((?:s_u32\(&sm\.)?(\w+)\)', code))
        for name in mapped:
            waits = re.findall(r"str_(?:wait|wait_peers|try_wait)\(&sm\.%s\b" % name, code)
            if waits:                                           # by a helper: the one whose instruction has the scope
                assert all(w.startswith("str_wait_peers") for w in waits), (path, name)
                body = code[code.index("bool str_try_wait_peers"):]
                assert "try_wait.parity.acquire.cluster" in body[:body.index("\n}\n")]
                assert "str_try_wait(" not in code[code.index("void str_wait_peers"):].split("\n}\n")[0]
            else:
                direct = re.findall(r'mbarrier\.try_wait\.([\w.:]*) p, \[%%1\][^"]*"[^;]*"r"\(%s\)' % name, code)
                assert direct and all("acquire.cluster" in d for d in direct), (path, name, direct)
            found += 1
    assert found >= 3


def test_a_running_maximum_is_one_value_for_a_warp():
    """What a warp reads of a word that others raise meanwhile is one lane's reading for all: its lanes would otherwise go by bounds
    of their own while one of them notes which batches a bound stands for."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "aq_attn.cu")).read())
    readings = re.findall(r"unsigned int (?:next|hint) = ([^;]*);", code)
    assert readings
    for r in readings:
        assert re.fullmatch(r"__shfl_sync\(0xFFFFFFFFu, .*, 0\)", r), r


@pytest.mark.gpu
@pytest.mark.parametrize("M,K", [(1, 32), (1, 64), (3, 32), (3, 96), (16, 4096), (17, 16384)])
def test_every_share_of_the_cluster_reaches_the_scale(M, K):
    """One value at a time carries the scale, from the first to the last share of a cluster; CTAs without a share of X are
    at the meeting at once. Codes and exponents as the checker's."""
    import oracle
    from gpu_util import dev, handle
    h = handle()
    for at in sorted({0, M * K - 1, *range(0, M * K, max(8, M * K // 16))}):
        x = np.full(M * K, 0.125, np.float16)
        x[at] = -37.5
        x = x.reshape(M, K)
        q, e = h.aq_quantize_act(dev(x), 8)
        assert int(e.item()) == oracle.layer_exponent(x, 8)
        assert np.array_equal(q.cpu().numpy(), oracle.quantize_act(x, 8, int(e.item())))
        qa, ea, zp = h.aq_quantize_act_asym(dev(x), 8)
        assert (int(ea.item()), int(zp.item())) == oracle.asym_params(x, 8)
