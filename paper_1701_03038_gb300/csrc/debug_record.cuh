// debug_record.cuh -- the records of the bounds-checked build, one for each
// source file with checks, read together.
#pragma once

namespace fstgpu {

// What a record holds: violations, and the first one's code, index and bound.
struct DebugCounts {
  unsigned long long violations = 0, code = 0, index = 0, bound = 0;
};

// A source file's record puts itself on the list that debug_read_all walks.
// `read` adds what it holds since the last read to *out and clears it
// (nonzero: an error).
struct DebugRecord {
  typedef int (*Read)(DebugCounts* out);
  Read read;
  DebugRecord* next;
  static DebugRecord*& list() {
    static DebugRecord* head = nullptr;
    return head;
  }
  explicit DebugRecord(Read r) : read(r), next(list()) { list() = this; }
};

// All records: the sum of their violations, and the first one found.
inline int debug_read_all(DebugCounts* out) {
  for (DebugRecord* r = DebugRecord::list(); r; r = r->next) {
    DebugCounts d;
    const int rc = r->read(&d);
    if (rc) return rc;
    if (d.violations && !out->violations) *out = d;
    else out->violations += d.violations;
  }
  return 0;
}

}  // namespace fstgpu
