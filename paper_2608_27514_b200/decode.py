"""Speculative decoding of one block as a sequence of libtsd calls (Alg. 1, Sections 3.1-3.3).

``BlockDecoder`` strings the library's kernels into the paper's loop.  One pass =

    caller's model forward over every node of the tree   (its attention layers call
                                                          ``VerifyStep.attention``)
    -> tsd_advance_block        scores of this pass = candidate pool of the next (Section 3.1), longest
                                verified trajectory (Section 3.3), next root into the token buffer with
                                its sequential step indices, tree of the next pass (Alg. 1 Phase 2)

All of it is enqueued on the current stream; the only thing that comes back per pass is the count of
rows still masked, which ends the loop: the pass writes it to pinned host memory (8 bytes per sequence)
and the loop watches that.  The class allocates and marshals;
every step of the arithmetic runs in the library's kernels.
"""
import torch

from . import binding as B


# Report words of decoders that are gone while a kernel may still have to write to them: the allocator of pinned memory knows
# nothing of that kernel and would give them to the next one who asks.  Given back once the words have arrived.
_unreported = {}


def _arrived(report, ticket):
    return bool((report >> 32 == ticket).all())


def _give_back():
    for key, words in list(_unreported.items()):
        if _arrived(*words):
            _unreported.pop(key, None)


class BlockDecoder:
    def __init__(self, step, width, depth, tau, mask_id, rule=B.TSD_ACCEPT_EXACT, search=B.TSD_SEARCH_GREEDY):
        """step: a VerifyStep whose layout (batch, branches, rows) fixes the tree size: every pass
        verifies step.B nodes per sequence (unused slots are copies of the root)."""
        self.step, self.width, self.depth, self.tau, self.mask_id = step, int(width), int(depth), float(tau), int(mask_id)
        self.rule, self.search = rule, search
        S, Bn, R, dev = step.S, step.B, step.R, step.device
        i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device=dev)
        # two copies of the tree: the builder reads the verified tree while it writes the next one
        self.trees = [dict(parent=i32(S, Bn), state=i32(S, Bn, R), prob=torch.zeros((S, Bn), device=dev),
                           n=i32(S)) for _ in range(2)]
        self.cur = 0
        self.root = i32(S, R)
        self.fill_step = i32(S, R)
        self.step_base = i32(S)
        self.n_masked = i32(S)
        _give_back()
        # words that the calls write a ticket to: the count of masked rows as soon as it is known, and behind all outputs
        self.report, self.done = torch.zeros((2, S), dtype=torch.int64, pin_memory=True)
        self.ticket = 0
        self.in_flight = None  # (words, ticket) that the last such call enqueued has yet to write, or None once seen
        self.begun = False  # the block has just begun, and that call has reported its masked rows
        self.n_forward = 0

    def __del__(self):
        words = getattr(self, "in_flight", None)
        if words and not _arrived(*words):
            _unreported[id(words)] = words

    @property
    def tree(self):
        return self.trees[self.cur]

    def start(self, root_state):
        """Begin a block from root_state int32 [S, R]; the first pass has no candidate pool yet, so
        its tree is the root alone (copies in the unused slots)."""
        st, t = self.step, self.tree
        if root_state.dim() != 2:
            raise IndexError("root_state is [sequences, rows]")
        root = root_state.to(device=st.device, dtype=torch.int32).expand(st.S, st.R).contiguous()
        # a captured call is replayed for as long as its graph lives, which this object knows nothing of: it reports nothing
        report = None if torch.cuda.is_current_stream_capturing() else self.report
        before = self.in_flight
        if report is not None:
            self._next_ticket(report)
        try:
            B.tsd_begin_block(root, self.mask_id, t["parent"], t["state"], t["n"], self.root, self.fill_step, self.step_base,
                              self.n_masked, report, self.ticket, st.status)
        except Exception:
            self.in_flight = before  # a call that is rejected writes nothing
            raise
        self.n_forward = 0
        self.begun = report is not None

    def advance(self, logits, tokens=None, block_start=None):
        """One pass after the caller's forward: logits [S*B*R, V] of the current tree's nodes."""
        self._advance(logits, tokens, block_start, None)

    def _advance(self, logits, tokens, block_start, report, done=None):
        st, t, nxt = self.step, self.tree, self.trees[1 - self.cur]
        if self.rule == B.TSD_ACCEPT_PROB and not hasattr(st, "draft_prob"):
            st.draft_prob = torch.empty((st.S, st.B, st.R), dtype=torch.float32, device=st.device)
        B.tsd_advance_block(logits, st.k, st.conf, st.topk_idx, st.topk_prob, st.lse, st.topk_ws, t["parent"], t["state"], self.mask_id,
                            self.tau, self.rule, self.search, st.edge_valid, st.prefix_len, st.accepted_node, st.accepted_len,
                            st.n_new_tokens, st.unmask_flag, st.unmask_tok, getattr(st, "draft_prob", None), tokens, block_start,
                            self.root, self.fill_step, self.step_base, self.n_masked, self.width, self.depth, nxt["parent"],
                            nxt["state"], nxt["prob"], nxt["n"], report, self.ticket, st.status, None, done)
        self.cur = 1 - self.cur
        self.n_forward += 1
        self.begun = False

    def _next_ticket(self, words=None):
        self.ticket = self.ticket % 0x7fffffff + 1
        if words is not None:
            self.in_flight = (words, self.ticket)

    def decode(self, forward, tokens=None, block_start=None, max_passes=None):
        """Run passes until no sequence has a masked row left.  forward(state int32 [S,B,R]) must
        return the logits [S*B*R, V] of every node (a device tensor the vocabulary pass accepts).  When it
        returns, all its outputs are complete, for the host and for any stream."""
        limit = self.step.R + 1 if max_passes is None else max_passes
        status = 1  # not known from a report
        if self.n_forward < limit:
            if not self.begun:
                self._next_ticket(self.report)
                B.tsd_report_block(self.n_masked, self.step.status, self.report, self.ticket)
            masked, status = B.tsd_wait_block(self.report, self.ticket)
            self.in_flight = None
            if masked == 0:
                status = 1
            while self.n_forward < limit and masked > 0:
                logits = forward(self.tree["state"])
                before = self.in_flight
                self._next_ticket(self.done)
                try:
                    self._advance(logits, tokens, block_start, self.report, self.done)
                except Exception:
                    self.in_flight = before
                    raise
                masked, status = B.tsd_wait_block(self.report, self.ticket)
            if self.in_flight is not None:
                B.tsd_wait_block(self.done, self.ticket)
                self.in_flight = None
        if status:
            self.step.check_status()
        return self.root
