"""Rules of the kernels that no run shows reliably when they are broken: checked on the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_05454_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".cu"))))
def test_read_only_loads_are_of_data_that_no_kernel_of_a_step_writes(name):
    """A kernel of a step may be resident while its predecessors still write.  A read-only load has no order against those
    writes, not even behind the wait, so it is for weights and tables: the rotary table (c4), the normalisation's gains (gr) and the embedding's rows (src)."""
    for m in re.finditer(r"__ldg\(\s*([A-Za-z_][\w.>-]*)", _source(name)):
        assert m.group(1) in ("c4", "gr", "src"), f"{name}: __ldg of {m.group(1)}"


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".cu"))))
def test_no_kernel_declares_data_of_the_step_read_only(name):
    """const T* __restrict__ lets the compiler choose the same read-only load by itself: for weights (embed, g, W0, W1) and for the
    lengths that the host copies before a plain launch (P, G)."""
    for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", _source(name)):
        assert m.group(1) in ("embed", "g", "W0", "W1", "P", "G"), f"{name}: {m.group(1)}"


TCGEN05 = ["gemm_stream.cuh", "gemm_pair.cuh", "attention_umma.cuh", "attention_rows.cuh"]


def _roles(name):
    """Set-up, roles (the branches on the warp behind the set-up's barrier; the last one with what follows them) of a tcgen05 kernel."""
    body = _source(name)
    at = body.index("tmem_base = *tmem_slot")
    return body[:at], re.split(r"\n  (?:if|\} else if) \(warp [^\n]*\) \{\n|\n  \} else \{\n", body[at:])


@pytest.mark.parametrize("name,n_roles", list(zip(TCGEN05, [4, 3, 4, 3])))
def test_no_role_starts_a_bounded_wait_before_the_preceding_kernel_has_ended(name, n_roles):
    """The limit of a wait is for this kernel's own copies and MMAs.  Every role (producers, issuers, epilogue or softmax) reaches
    pdl_wait(), whatever early says, before its first mbar_wait()."""
    setup, (ahead, *roles) = _roles(name)
    roles = [r for r in roles if "mbar_wait(" in r]
    assert len(roles) == n_roles
    assert "mbar_wait(" not in ahead and "mbar_wait(" not in setup[setup.index("__global__"):]
    for r in roles:
        assert re.search(r"^ +pdl_wait\(\);", r.split("mbar_wait(")[0], re.M)


@pytest.mark.parametrize("name", ["gemm_stream.cuh", "gemm_pair.cuh"])
def test_a_rotary_projection_releases_the_attention_behind_its_own_wait(name):
    """The attention reads the descriptor and older cache rows ahead of its wait: the projection before it must not let it start until
    everything older has ended."""
    body = _source(name)
    assert [m.group(0) for m in re.finditer(r"[^\n]*pdl_release\(\);", body)] == ["  if (!kRope) pdl_release();", "    if (kRope) pdl_release();"]
    assert re.search(r"\n    pdl_wait\(\);\s*\n    if \(kRope\) pdl_release\(\);", body)


@pytest.mark.parametrize("name", ["attention_umma.cuh", "attention_rows.cuh"])
def test_attention_reads_only_older_rows_ahead_of_its_wait(name):
    """Ahead of the wait: nothing but the descriptor, and K / V tiles of cache rows that this pass's projection does not write (in place:
    those that end ahead of the pass's first row)."""
    _, (ahead, *roles) = _roles(name)
    assert "if (!early) pdl_wait();" in ahead
    assert len(re.findall(r"__ldcg\(sd\.\w+ \+ b(?: \+ 1)?\)", ahead)) == len(re.findall(r"\bsd\.", ahead)) == 3      # past L1
    copies = [r for r in roles if re.search(r"tma_load|load_tile\(", r)]
    assert len(copies) == 1
    early = copies[0].split("pdl_wait();")[0]
    loads = early[early.index("int issued = 0;"):]
    assert re.search(r"if \(early\)\s+while \(issued < min\(2, n_tiles\) && \(inplace \? [^?]*\* AU_BN <= F - Qn : [^?]* < n_c\)\) "
                     r"load_tile\(issued\+\+\);\s*$", loads)
    assert "load_tile(" not in early[:early.index("auto load_tile")]


def test_attention_starts_early_only_behind_a_rotary_projection_that_was_launched():
    """Which kernel ran decides, not which one was asked for."""
    src = _source("lsp_api.cu")
    assert re.findall(r"rotary_late = ([^;]+);", src) == ["0", "0", "std::is_same<Epi, EpiQKVRope<bf16>>::value ? 1 : 0"]
    last = re.findall(r"run_attention<\w+>\(.*, ([^,\n]+)\)[;\n]", src)
    assert last == ["c->rotary_late", "0", "0"]


@pytest.mark.parametrize("name", TCGEN05)
def test_warps_leave_on_an_expired_wait_as_one(name):
    """Tensor-memory loads and full-mask barriers need every lane: whether a wait expired is put to a vote before anyone leaves."""
    assert not re.search(r"if \(!mbar_wait\(", _source(name))


@pytest.mark.parametrize("name,warps", [("gemm_stream.cuh", [0, 6]), ("gemm_pair.cuh", [0])])
def test_producers_that_share_a_stage_outstay_their_copies_after_a_failure(name, warps):
    """A stage's barrier counts the copies of two producers (the weights' and the activations' warp, the two CTAs of a pair).  One that gives
    up leaves the other's copies on a barrier that never completes, so after a failure every warp that issues copies stays for a time."""
    body = _source(name)
    body = body[body.index("tmem_base = *tmem_slot"):]
    roles = re.split(r"\n  (?:if|\} else if) \(warp == ([^\n]*)\) \{\n|\n  \} else \{\n", body)
    issuing = [int(w) for w, r in zip(roles[1::2], roles[2::2]) if re.search(r"request_weights\(|load_weights\(|load_acts\(", r)]
    assert issuing == warps
    if len(warps) == 1:
        assert "if (!ok) um_let_land();" in roles[2]
        return
    for w, r in zip(roles[1::2], roles[2::2]):
        if w in map(str, warps):          # every wait of such a warp that expires
            waits = re.split(r"if \(!__all_sync\(0xffffffffu, mbar_wait\(|&& !__all_sync\(0xffffffffu, mbar_wait\(", r)[1:]
            assert len(waits) == (2 if w == "0" else 1) == r.count("mbar_wait(")
            assert all(re.search(r"um_let_land\(\);\s*break;", x) for x in waits)


def test_the_paired_gemm_models_the_tiles_that_it_launches():
    """The choice of a tile width and the launch count column tiles by one function (rotary tiles of several heads come in twos)."""
    src = _source("gemm_pair.cuh")
    assert re.findall(r"[^\n]*pair_tiles\([^\n]*", src) == [
        "inline int pair_tiles(int cols, int bn, int rot_half) {",
        "    const long t = (long)pair_tiles(cols, bn, rot_half) * rg;",
        "  const int n_tiles = pair_tiles(cols, bn, rot_half);"]


def test_the_step_driver_assumes_no_sm_count():
    """The dispatch lines of the CUDA-core kernels (fp32 models among them) are in SMs of the device at hand."""
    assert not re.search(r"\b148\b", _source("lsp_api.cu")) and "cudaDevAttrMultiProcessorCount" in _source("lsp_api.cu")
