"""Kernels launched programmatically overlap their predecessor, which may still be
writing the stream's vectors and scalars when they start.  Data that changes
during a kernel must not be read as read-only data (ld.global.nc, __ldg, or a
const __restrict__ pointer, which the compiler may turn into such loads).  This
reads the sources: in every kernel that waits for its predecessor, and in every
function it calls, only matrices, scalings fixed at setup and launch descriptors
are read that way."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_05686_gb300", "csrc")
FILES = ["common.cuh", "reduce.cuh", "solve.cuh", "vkern.cuh", "group.cuh", "solve.cu", "vcycle.cu", "block.cu",
         "dense.cu", "group.cu"]
# matrix arrays, D^-1/2 and sqrt(diag) (written at setup)
MATRIX = {("int64_t", "rp"), ("int64_t", "sp"), ("int32_t", "ci"), ("int32_t", "base"), ("uint16_t", "c16"),
          ("T", "v"), ("double", "v"), ("double", "s"), ("double", "sq")}
# written by a copy before the launches that read them
DESCRIPTORS = {"D", "GMat<T>", "GVec<T>", "GCg", "CoarseEnt", "CoarseProb"}


def functions():
    """name -> (file, parameter list, body) of every device function"""
    out = {}
    for f in FILES:
        s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        s = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", s)
        for m in re.finditer(r"__(?:global|device)__[^;{}()=]*?\b(\w+)\s*\(", s):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(s[i], 0)
                i += 1
            par = s[m.end():i - 1]
            rest = s[i:].lstrip()
            if not rest.startswith("{"):
                continue
            b = s.index("{", i)
            e, depth = b + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(s[e], 0)
                e += 1
            out.setdefault(m.group(1), []).append((f, m.group(0), par, s[b:e]))
    return out


def closure(fs):
    """kernels that reach pdl_sync, and all that they call"""
    calls = {n: {k for k in fs if any(re.search(rf"\b{k}\b", body) for *_, body in defs)} for n, defs in fs.items()}

    def reach(n, seen):
        if n not in seen:
            seen.add(n)
            for k in calls[n]:
                reach(k, seen)
        return seen
    kernels = [n for n, defs in fs.items() if any("__global__" in h for _, h, *_ in defs)]
    waiting = [n for n in kernels if "pdl_sync" in reach(n, set())]
    return waiting, set().union(*(reach(n, set()) for n in waiting))


def test_overlapping_kernels_read_vectors_with_plain_loads():
    fs = functions()
    waiting, names = closure(fs)
    assert {"k_vc_cheb", "k_bvc_cheb", "k_dots", "k_cg_update", "k_bcg_pupdate", "k_power_prep", "k_fin_wide",
            "k_coarse", "k_g_mat", "k_g_cg_rows", "k_bsell_spmv_dot"} <= set(waiting)
    assert {"row_apply_at", "brow_apply", "sell_row", "csr_lane", "ldvec", "coarse_rows"} <= names
    bad = []
    for n in sorted(names):
        for f, _, par, body in fs[n]:
            if re.search(r"__ldg\s*\(|ld\.global\.nc", body):
                bad.append(f"{f}: {n} reads with __ldg or ld.global.nc")
            for t, p in re.findall(r"const\s+([\w<>:]+)\s*\*\s*__restrict__\s+(\w+)", par):
                if (t, p) not in MATRIX and t not in DESCRIPTORS:
                    bad.append(f"{f}: {n}: const {t}* __restrict__ {p}")
            for t, p, v in re.findall(r"const\s+([\w<>:]+)\s*\*\s*__restrict__\s+(\w+)\s*=\s*([^;]*);", body):
                if not re.match(r"M\.(v|ci)\b|M \+", v):
                    bad.append(f"{f}: {n}: local const {t}* __restrict__ {p}")
    assert not bad, "\n".join(bad)


def test_waits_acquire_what_they_wait_for():
    """a wait on a flag that announces data acquires it, and the flag is released:
    a volatile access orders nothing after it"""
    fs = functions()
    for name, order in (("potrf_inv", "cta"), ("ch_poll", "gpu"), ("ch_publish", "gpu")):
        (_, _, _, body), = fs[name]
        text = body + "".join(b for k in ("cta_release", "cta_acquire") if re.search(rf"\b{k}\b", body)
                              for *_, b in fs.get(k, ()))
        assert re.search(rf"(st\.release|ld\.acquire)\.{order}\.", text), name
        if name == "potrf_inv":
            assert "volatile int" not in text and f"st.release.{order}.shared" in text
            assert f"ld.acquire.{order}.shared" in text
